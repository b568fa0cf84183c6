// Many time steps of one small lattice in one launch, its populations
// resident in shared memory (FP32-deviation and FP64 storage, MRT or BGK, at
// most one body of any shape and motion, every boundary kind).
//
// What bounds it.  A lattice of up to half a million nodes fits the shared
// memory of the chip, so HBM does not bound its steps; launched step by step
// it was bound by the launch boundary and by the chain of memory round trips
// of a step (9 to 14 us whatever the size).  Here one block per SM owns a
// rectangle of nodes for up to RES_MAX_STEPS steps.  A step costs a block
// its node updates (registers and shared memory only) and one exchange of
// the three outward populations of each edge node with its eight neighbours.
//
// Exchange.  Every 32-bit word crosses L2 as one 64-bit word {value, tag}:
// a 64-bit element of an access is not torn, so a receiver that reads the tag
// of this step has the value of this step, and the exchange needs no fence and
// no flag, one L2 trip per step.  The tag counts steps over all launches of
// the context.  A trip takes 600 clocks on one die and 1 100 to the other if
// sender and receiver use one access each; several coherent loads of one
// thread follow one another (eight: 3 000 clocks), so every word here is laid
// out for one 16-byte access per thread.  Mailboxes alternate with the step
// parity: a block writes step n's words only after it read its neighbours'
// words of step n - 1, which they sent after reading its words of step n - 2,
// so a word is read before it is overwritten.
//
// Tiles.  A block is 512 threads; a thread owns K nodes (K = 1 .. 7 fixed
// at compile time, node t, t + 512, ...).  A step pulls the K nodes' nine
// populations from the stage into registers, meets the block, updates and
// overwrites them: one stage, not two, so that 1230 x 410 fits.  The nodes
// inside a tile are pulled while the neighbours' words are on their way; the
// tile's edge nodes come first in the order, so their words leave while the
// rest is updated, and the boundary rules of lattice-edge nodes are evaluated
// once per launch (edge_pull).  A node's nine populations are adjacent in the
// stage (stride 9: conflict-free).  The update is the one-step kernels' code
// (FP32 MRT on paired lanes, two of the thread's nodes at a time), so the
// populations are those kernels' bit for bit.
//
// Body.  One more block (the tail) publishes the pose of every step in a
// ring of tagged words, gathers the partial sums of the tiles that meet the
// body and writes the records (Eqs. 25-27).  On a prescribed path its eight
// warps take every eighth step each, so a pose is out eight steps before it
// is used; for a free body one warp sums the forces, advances the body
// (Eqs. 23-24) and publishes the next pose, which the tiles wait for.  The
// tiles that meet the body sum the momentum exchanged before their update,
// and the penalization's reaction behind it.
//
// Every wait is bounded (ResidentLaunch::timeout_ns): a thread whose wait
// gives up latches ERR_TIMEOUT and its block leaves; the others' waits then
// run out likewise.  The launch is cooperative: all blocks are resident.
//
// Measured (GB300, us per step, one-step launches -> this kernel): FP32 256 x
// 128 with a fixed disk 8.9 -> 2.4, 512 x 256 oscillating disk 8.7 -> 2.8, 512
// x 256 disk on a spring (free) 14.1 -> 4.7, 700 x 400 9.0 -> 4.3, 1230 x 410
// 10.5 -> 6.2; FP64 256 x 128 13.6 -> 6.5 (8.1 with the solid-node sums in FP64
// instructions).  What is left: the update itself at
// 7 nodes a thread (issue slots about half busy), and below 2 nodes a thread
// the exchange and the three block barriers of a step.  Contexts on streams of
// their own gain less, since a launch takes every SM (resident_now, capi.cu).
#define VPLBM_PLAIN_LOADS 1
#include "vplbm_node.cuh"

namespace vplbm {
namespace {

// Threads of a block.  128 registers a thread hold seven FP32 nodes and one
// update without spilling; more threads with fewer nodes each were slower
// (1230 x 410, us per step: 512 x 7 nodes 6.0, 640 x 6 7.2, 896 x 4 8.0).
constexpr int RES_NT = 512;
constexpr int RES_RECV = 2;          // 16-byte mailbox accesses a thread makes per step at most
constexpr int RES_TAIL_WARPS = 8;    // steps the tail works on at a time (prescribed path)
constexpr int POSE_WORDS = (int)(sizeof(BodyState) / 4);

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void send_word(uint64_t *p, uint32_t v, uint32_t tag)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((uint64_t)tag << 32) | v) : "memory");
}

// The bound of a wait: counts polls, and looks at the timer now and then.
struct Patience {
    unsigned long long t0 = 0;
    unsigned n = 0;
    __device__ __forceinline__ bool out(unsigned long long limit)
    {
        if ((++n & 255u) != 0) return false;
        const unsigned long long t = global_ns();
        if (t0 == 0) t0 = t;
        return t - t0 > limit;
    }
};

// Two words at a 16-byte boundary in one access.
struct Pair {
    uint64_t a, b;
    __device__ __forceinline__ bool both(uint32_t tag) const { return (uint32_t)(a >> 32) == tag && (uint32_t)(b >> 32) == tag; }
};
__device__ __forceinline__ void send_pair(uint64_t *p, uint32_t v, uint32_t w, uint32_t tag)
{
    const uint64_t t = (uint64_t)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | v), "l"(t | w) : "memory");
}
__device__ __forceinline__ Pair read_pair(const uint64_t *p)
{
    Pair r;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(r.a), "=l"(r.b) : "l"(p) : "memory");
    return r;
}

// Both words of tag `tag` into r (looked at first as it is); false if the wait
// gave up.
__device__ __forceinline__ bool wait_pair(const ResidentLaunch &L, const uint64_t *p, uint32_t tag, Pair &r)
{
    Patience pt;
    while (!r.both(tag)) {
        if (pt.out(L.timeout_ns)) {
            atomicOr(L.p.err, ERR_TIMEOUT);
            return false;
        }
        r = read_pair(p);
    }
    return true;
}

__device__ __forceinline__ uint64_t *pose_slot(const ResidentLaunch &L, int k)
{
    return L.poses + (size_t)(k % L.t.pose_ring) * POSE_WORDS;
}

// Partial sums of the tiles that meet the body, slot by slot: the forces (and
// the node count) for reader r, the penalization's reaction.  A free body's
// forces are waited for, by the tail (r = 0) and by each of those tiles (r = 1
// + slot): each has a copy of its own, written in one transaction, since
// several tiles polling the L2 lines that several others still write took 9 k
// clocks per message instead of 3 k.
__device__ __forceinline__ uint64_t *force_slot(const ResidentLaunch &L, int k, int slot, int r)
{
    return L.parts + (((size_t)(k % RES_PART_RING) * L.t.part_copies + r) * L.t.part_slots + slot) * 8;
}
__device__ __forceinline__ uint64_t *react_slot(const ResidentLaunch &L, int k, int slot)
{
    return L.parts + ((size_t)RES_PART_RING * L.t.part_copies + (size_t)(k % RES_PART_RING)) * L.t.part_slots * 8 + (size_t)slot * 8;
}

// Tiles that meet the body's node range: first column and row, columns and
// rows; tile (0, 0) stands in for an empty range.
__device__ __forceinline__ int4 tile_rect(const ResidentPlan &t, const int4 range, int nx, int ny)
{
    if (range.x > range.y) return make_int4(0, 0, 1, 1);
    // column c holds nodes [c nx / ntx, (c + 1) nx / ntx)
    const int c0 = ((range.x + 1) * t.ntx - 1) / nx, c1 = ((range.y + 1) * t.ntx - 1) / nx;
    const int r0 = ((range.z + 1) * t.nty - 1) / ny, r1 = ((range.w + 1) * t.nty - 1) / ny;
    return make_int4(c0, r0, c1 - c0 + 1, r1 - r0 + 1);
}

// A published pose carries its tile rectangle in the padding of BodyState
// (pad0: first column and row, pad: columns and rows), so that the tiles do
// not divide for it every step.
__device__ __forceinline__ int set_rect(const ResidentLaunch &L, BodyState *bs)
{
    const int4 r = tile_rect(L.t, make_int4(bs->ilo, bs->ihi, bs->jlo, bs->jhi), L.p.nx, L.p.ny);
    bs->pad0 = (long long)(((uint64_t)(uint32_t)r.y << 32) | (uint32_t)r.x);
    bs->pad[0] = r.z;
    bs->pad[1] = r.w;
    return r.z * r.w;
}
__device__ __forceinline__ BodyState without_rect(BodyState s)
{
    s.pad0 = 0;
    s.pad[0] = s.pad[1] = 0;
    return s;
}

// ---- the tail block ----------------------------------------------------

// Sum over step k's partials at `from`, np slots of four sums: lane 4 s + q
// takes sum q of the slots s, s + 8, ..., then the lanes of a sum are added (a
// fixed order).  Lane q < 4 returns sum q.
template <typename A>
__device__ __forceinline__ bool gather_parts(const ResidentLaunch &L, int k, int np, const uint64_t *from, A &sum)
{
    const int lane = threadIdx.x & 31;
    const uint32_t tag = L.tag0 + (uint32_t)k;
    bool ok = true;
    acc_zero(sum);
    for (int s = lane >> 2; s < np && ok; s += 8) {
        const uint64_t *at = from + (size_t)s * 8 + 2 * (lane & 3);
        Pair r = read_pair(at);
        ok = wait_pair(L, at, tag, r);
        const uint32_t w0 = (uint32_t)r.a, w1 = (uint32_t)r.b;
        if constexpr (sizeof(typename SumVal<A>::V) == 8)
            acc_add(sum, __longlong_as_double((long long)(((uint64_t)w1 << 32) | w0)));
        else
            acc_add(sum, make_float2(__uint_as_float(w0), __uint_as_float(w1)));
    }
    if (!__all_sync(0xffffffffu, ok)) return false;
    for (int off = 16; off >= 4; off >>= 1)
        if (off < 4 * np) acc_add(sum, acc_shfl_down(sum, off));   // uniform: the lanes from 4 np on hold zeros
    return true;
}

// floor and ceil of a double of magnitude below 2^30, and its fraction
// (d - floor(d), d >= 2^-11, rounded to FP32), on the integer pipe.
__device__ __forceinline__ int int_floor(double d, bool up)
{
    const uint64_t b = (uint64_t)__double_as_longlong(d);
    const int e = (int)((b >> 52) & 0x7ff) - 1023;
    const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);
    const int ip = e < 0 ? 0 : (int)(m >> (52 - e));
    const bool rest = e < 0 ? (b << 1) != 0 : (m << (12 + e)) != 0;
    const bool neg = (long long)b < 0;
    return (neg ? -ip : ip) + (rest && neg != up ? (up ? 1 : -1) : 0);
}
__device__ __forceinline__ float fraction(double d)
{
    const uint64_t b = (uint64_t)__double_as_longlong(d);
    const int e = (int)((b >> 52) & 0x7ff) - 1023;
    const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);
    return (float)(m << (12 + e)) * 0x1p-64f;
}

// The free body's next pose from the force of this step (Algorithm 1, step
// 3), lane d < 3 its degree of freedom d.  This is the critical path of a
// free body's step, and an FP64 instruction costs a warp 65 clocks on GB300,
// dependent or not, so it is built from few of them.  RK4 of m q'' + c q' +
// k (q - q0) = F, F held over the step, is an affine map of (q, v): with
// A = F - c v - k (q - q0),  q += P11 v + P12 A,  v += P21 v + P22 A, where
// P = I + L / 2 + L^2 / 6 + L^3 / 24, L = [[0, 1], [-k/m, -c/m]]
// (ResidentLaunch::rk; P12 and P22 over m).  The values derived from the pose
// are derive_pose's, by integer arithmetic.
struct FreeBody {   // a lane's degree of freedom
    double f_ext, damp, stiff, q0, p11, p12, p21, p22, radius;
    bool on, disk;
    int n;          // nodes along its axis
};
__device__ __forceinline__ FreeBody free_body(const ResidentLaunch &L)
{
    const int lane = threadIdx.x & 31, d = lane < 3 ? lane : 0;
    const DevBody &b = L.p.body;
    return {b.f_ext[d], b.damp[d], b.stiff[d], b.q0[d], L.rk[d][0], L.rk[d][1], L.rk[d][2], L.rk[d][3], b.radius,
            ((b.dof_mask >> d) & 1u) != 0, b.shape == VPLBM_SHAPE_DISK, d == 0 ? L.p.nx : L.p.ny};
}

__device__ __forceinline__ void advance_free(const ResidentLaunch &L, const FreeBody &b, BodyState *bs, double F)
{
    const StepParams &p = L.p;
    const int lane = threadIdx.x & 31, d = lane < 3 ? lane : 0;
    double q = bs->q[d], v = bs->v[d];
    const double A = F + b.f_ext - b.damp * v - b.stiff * (q - b.q0);
    if (b.on) {
        q = fma(b.p12, A, fma(b.p11, v, q));
        v = fma(b.p22, A, fma(b.p21, v, v));
    }
    const double lo = q - b.radius, hi = q + b.radius;
    __syncwarp();
    // ordinary poses (1 <= q, all below 2^29 in magnitude); elsewhere (left of
    // or below the lattice's first nodes, far away, not finite) derive_pose
    // itself
    const int el = (__double2hiint(lo) >> 20) & 0x7ff, eh = (__double2hiint(hi) >> 20) & 0x7ff, eq = __double2hiint(q) >> 20;
    const bool plain = b.disk && el < 1023 + 29 && eh < 1023 + 29 && eq >= 1023 && eq < 1023 + 29;
    if ((__ballot_sync(0xffffffffu, plain) & 3u) == 3u) {
        const int l = max(int_floor(lo, false) - 1, 0), h = min(int_floor(hi, true) + 1, b.n - 1);
        const bool in = (__ballot_sync(0xffffffffu, l <= h) & 3u) == 3u;
        if (lane < 2) {
            (lane ? bs->jlo : bs->ilo) = in ? l : 1;
            (lane ? bs->jhi : bs->ihi) = in ? h : 0;
            (lane ? bs->yi : bs->xi) = in ? int_floor(q, false) : 0;
            (lane ? bs->yf : bs->xf) = in ? fraction(q) : 0.f;
        }
        if (lane < 3) {
            bs->q[d] = q;
            bs->v[d] = v;
            (d == 0 ? bs->vxf : d == 1 ? bs->vyf : bs->omf) = (float)v;
        }
        if (lane == 0) bs->step += 1;
    } else {
        if (lane < 3) {
            bs->q[d] = q;
            bs->v[d] = v;
        }
        __syncwarp();
        if (lane == 0) {
            BodyState s = *bs;
            s.step += 1;
            derive_pose(s, p.body.present, p.body.radius, p.nx, p.ny, p.body.shape);
            *bs = s;
        }
    }
    __syncwarp();
    {   // set_rect, a division per lane
        const int m = lane & 3, at = (&bs->ilo)[m];   // ilo, ihi, jlo, jhi
        const int div = m < 2 ? ((at + 1) * L.t.ntx - 1) / p.nx : ((at + 1) * L.t.nty - 1) / p.ny;
        const int c1 = __shfl_sync(0xffffffffu, div, 1), r0 = __shfl_sync(0xffffffffu, div, 2), r1 = __shfl_sync(0xffffffffu, div, 3);
        if (lane == 0) {
            const bool any = bs->ilo <= bs->ihi;
            bs->pad0 = any ? (long long)(((uint64_t)(uint32_t)r0 << 32) | (uint32_t)div) : 0;
            bs->pad[0] = any ? c1 - div + 1 : 1;
            bs->pad[1] = any ? r1 - r0 + 1 : 1;
        }
    }
    __syncwarp();
}

// *bs := pose k + 1, from pose k and the forces of the tiles that meet it.
// Every warp that does this (the tail's, one in each of those tiles) has the
// same pose: the same sums in the same order.
template <typename A>
__device__ __forceinline__ bool next_pose(const ResidentLaunch &L, int k, const FreeBody &fb, BodyState *bs, int r)
{
    A F;   // lane d < 3: of degree of freedom d
    if (!gather_parts<A>(L, k, bs->pad[0] * bs->pad[1], force_slot(L, k, 0, r), F)) return false;
    advance_free(L, fb, bs, acc_value(F));
    return true;
}

// A tile that meets a free body: pose k + 1 into s_bs[(k + 1) & 1] by one of
// its warps.
template <typename A>
__device__ __noinline__ bool tile_next_pose(const ResidentLaunch &L, int k, BodyState *s_bs, int slot)
{
    const int lane = threadIdx.x & 31;
    const BodyState *now = s_bs + (k & 1);
    BodyState *next = s_bs + ((k + 1) & 1);
    // not more than 4 steps ahead of the tail, whose warps read the partials too
    // (at most 8 steps behind its first)
    Pair w{0, 0};
    const uint64_t *at = pose_slot(L, k - 4);
    if (k >= 4) w = read_pair(at);
    for (int m = lane; m < POSE_WORDS; m += 32)
        reinterpret_cast<uint32_t *>(next)[m] = reinterpret_cast<const uint32_t *>(now)[m];
    __syncwarp();
    if (!next_pose<A>(L, k, free_body(L), next, 1 + slot)) return false;
    return k < 4 || wait_pair(L, at, L.tag0 + (uint32_t)(k - 4), w);
}

__device__ __forceinline__ void publish_pose(const ResidentLaunch &L, int k, const BodyState *bs)
{
    const int lane = threadIdx.x & 31;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(bs);
    uint64_t *dst = pose_slot(L, k);
    if (lane < POSE_WORDS / 2) send_pair(dst + 2 * lane, src[2 * lane], src[2 * lane + 1], L.tag0 + (uint32_t)k);
}

// Step k's record: gathers its sums (one warp).
template <typename A>
__device__ __forceinline__ bool write_record(const ResidentLaunch &L, int k, const BodyState &bs)
{
    const StepParams &p = L.p;
    const int np = bs.pad[0] * bs.pad[1];
    A force, react;
    if (!gather_parts<A>(L, k, np, force_slot(L, k, 0, 0), force) || !gather_parts<A>(L, k, np, react_slot(L, k, 0), react))
        return false;
    if ((long long)k + p.hist_cap < L.nsteps) return true;   // overwritten later in this launch
    const double f = acc_value(force), r = acc_value(react);
    double sum[NPART - 1];
#pragma unroll
    for (int q = 0; q < 3; ++q) sum[q] = __shfl_sync(0xffffffffu, r, q);
#pragma unroll
    for (int q = 0; q < 4; ++q) sum[3 + q] = __shfl_sync(0xffffffffu, f, q);
    if ((threadIdx.x & 31) != 0) return true;
    vplbm_record rec;
    rec.t = (double)bs.step;
    rec.fx = sum[3]; rec.fy = sum[4]; rec.torque = sum[5];
    rec.cd = sum[3] * p.body.inv_qref;
    rec.cl = sum[4] * p.body.inv_qref;
    rec.x = bs.q[0]; rec.y = bs.q[1]; rec.theta = bs.q[2];
    rec.vx = bs.v[0]; rec.vy = bs.v[1]; rec.omega = bs.v[2];
    rec.fpen_x = sum[0]; rec.fpen_y = sum[1]; rec.tpen = sum[2];
    rec.n_solid = sum[6];
    p.hist[bs.step % p.hist_cap] = rec;
    return true;
}

template <int P>
__device__ __noinline__ void resident_tail(const ResidentLaunch &L, BodyState *s_bs)
{
    using A = typename SumT<P>::A;
    const StepParams &p = L.p;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const BodyState start = *p.bs_in;
    if (threadIdx.x == 0) s_bs[RES_TAIL_WARPS].ilo = s_bs[RES_TAIL_WARPS].ihi = s_bs[RES_TAIL_WARPS].jlo = 0;
    __syncthreads();   // bs_out may be the same slot
    if (warp >= RES_TAIL_WARPS) return;
    BodyState *bs = s_bs + warp;
    if (prescribed_motion(p)) {
        // warp w: steps w, w + 8, ...; index nsteps is the pose the next launch starts from
        for (int k = warp; k <= L.nsteps; k += RES_TAIL_WARPS) {
            if (lane == 0) {
                BodyState s = start;
                const double F0[3] = {0.0, 0.0, 0.0};
                if (k > 0) {   // a prescribed pose depends on its step alone
                    const long long at = s.step + k;
                    body_advance(p.body, at - 1, F0, s.q, s.v);
                    s.step = at;
                    derive_pose(s, p.body.present, p.body.radius, p.nx, p.ny, p.body.shape);
                }
                if (k == L.nsteps) *L.bs_out = s;
                set_rect(L, &s);
                *bs = s;
            }
            __syncwarp();
            if (k == L.nsteps) break;
            publish_pose(L, k, bs);
            if (!write_record<A>(L, k, *bs)) return;
            __syncwarp();
        }
        return;
    }
    // a free body: warp 0 advances the body for the tiles that do not meet it
    // (those that do advance it themselves), warps 1 and 2 write the records
    // of every other step behind it
    volatile int *done = &s_bs[RES_TAIL_WARPS].ilo;   // records written by warp 1, 2
    if (warp == 0) {
        const FreeBody fb = free_body(L);
        if (lane == 0) {
            *bs = start;
            set_rect(L, bs);
        }
        __syncwarp();
        publish_pose(L, 0, bs);
        for (int k = 0; k < L.nsteps; ++k) {
            // the records' warps read the partials of the last few steps
            bool ok = true;
            Patience pt;
            while (k - 2 * min(done[0], done[1]) > RES_PART_RING / 2 && ok) ok = !pt.out(L.timeout_ns);
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
                return;
            }
            if (!next_pose<A>(L, k, fb, bs, 0)) return;
            if (k + 1 < L.nsteps) publish_pose(L, k + 1, bs);
        }
        if (lane == 0) *L.bs_out = without_rect(*bs);
    } else if (warp <= 2) {
        for (int k = warp - 1; k < L.nsteps; k += 2) {
            bool ok = true;
            if (lane < POSE_WORDS / 2) {
                const uint64_t *at = pose_slot(L, k) + 2 * lane;
                Pair r = read_pair(at);
                ok = wait_pair(L, at, L.tag0 + (uint32_t)k, r);
                reinterpret_cast<uint2 *>(bs)[lane] = make_uint2((uint32_t)r.a, (uint32_t)r.b);
            }
            if (!__all_sync(0xffffffffu, ok)) return;
            __syncwarp();
            if (!write_record<A>(L, k, *bs)) return;
            if (lane == 0) done[warp - 1] = k / 2 + 1;
            __syncwarp();
        }
        if (lane == 0) done[warp - 1] = L.nsteps;
    }
}

// ---- the tiles ---------------------------------------------------------

// An exact sum of 64-bit fixed-point terms (FP64 storage, MRT: the solid-node
// sums of a tile, since an FP64 addition costs a warp 65 clocks): the terms'
// high words and their low words, summed apart.
struct FxSum {
    long long hi, lo;
};
__device__ __forceinline__ void acc_zero(FxSum &a) { a.hi = a.lo = 0; }
__device__ __forceinline__ void acc_add(FxSum &a, FxSum b)
{
    a.hi += b.hi;
    a.lo += b.lo;
}
__device__ __forceinline__ FxSum acc_shfl_down(FxSum a, int off)
{
    return {__shfl_down_sync(0xffffffffu, a.hi, off), __shfl_down_sync(0xffffffffu, a.lo, off)};
}
__device__ __forceinline__ FxSum fx_term(long long x) { return {x >> 32, (long long)(uint32_t)(uint64_t)x}; }
// x y, y an int of up to 12 bits.
__device__ __forceinline__ FxSum fx_term(long long x, int y) { return {(x >> 32) * y, (long long)(uint32_t)(uint64_t)x * y}; }
// The sum in units of 2^k, as a double.
__device__ __forceinline__ double fx_value(FxSum a, int k)
{
    const long long hi = a.hi + (a.lo >> 32);
    if (hi + (1LL << 30) >= 0 && hi < 1LL << 30) return fx_signed_to((long long)((uint64_t)hi << 32) + (long long)(uint32_t)(uint64_t)a.lo, k);
    return ((double)hi * 4294967296.0 + (double)(uint32_t)(uint64_t)a.lo) * ldexp(1.0, k);
}

// A node's word: its column (bits 0-11) and row (12-23) in the tile, and
constexpr unsigned ND_VALID = 1u << 24, ND_LATTICE_EDGE = 1u << 25, ND_EDGE = 1u << 26, ND_CORNER = 1u << 27;
__device__ __forceinline__ int nd_x(unsigned b) { return (int)(b & 0xfffu); }
__device__ __forceinline__ int nd_y(unsigned b) { return (int)((b >> 12) & 0xfffu); }
__device__ __forceinline__ int nd_off(unsigned b, int pitch) { return ((nd_y(b) + 1) * pitch + nd_x(b) + 1) * NQ; }

// The pull of population a into lattice-edge node (i, j) of a tile, as data:
// the boundary rules (pull_edge_src) are evaluated once per launch, and a
// step's pull is a load, for a moving wall an addition, for the convective
// outlet its mix.  at: the place in the stage that is read (a node reached
// across a periodic edge sits at its unwrapped place, in the ring) and how.
constexpr unsigned EDGE_ADD = 1u << 30, EDGE_OUTLET = 1u << 31;
template <typename T> struct EdgePull {
    unsigned at;
    T cu;   // c_a . u_w of a moving wall
};
template <typename T> __device__ __forceinline__ T wall_cu(const StepParams &p, int a, int side, int k);
template <> __device__ __forceinline__ double wall_cu<double>(const StepParams &p, int a, int side, int k)
{
    return cx_of(a) * wall_u(p, side, 0, k) + cy_of(a) * wall_u(p, side, 1, k);
}
template <> __device__ __forceinline__ float wall_cu<float>(const StepParams &p, int a, int side, int k)
{
    return (float)cx_of(a) * wall_uf(p, side, 0, k) + (float)cy_of(a) * wall_uf(p, side, 1, k);
}
template <typename T>
__device__ __forceinline__ EdgePull<T> edge_pull(const StepParams &p, int a, int i, int j, int i0, int j0, int pitch)
{
    auto place = [&](int b, int x, int y) { return (unsigned)(((y - j0 + 1) * pitch + x - i0 + 1) * NQ + b); };
    const int si = i - cx_of(a), sj = j - cy_of(a);
    if (sj < 0 || sj >= p.ny) {
        const int side = sj < 0 ? VPLBM_SOUTH : VPLBM_NORTH, kind = p.bc[side];
        if (kind == VPLBM_BC_SYMMETRY) {
            const bool out = (si < 0 || si >= p.nx) && p.bc[VPLBM_WEST] != VPLBM_BC_PERIODIC;
            return {place(miry_of(a), out ? i : si, j), (T)0};
        }
        if (kind == VPLBM_BC_VELOCITY) return {place(opp_of(a), i, j) | EDGE_ADD, wall_cu<T>(p, a, side, i)};
        if (kind != VPLBM_BC_PERIODIC) return {place(opp_of(a), i, j), (T)0};
    }
    if (si < 0 || si >= p.nx) {
        const int side = si < 0 ? VPLBM_WEST : VPLBM_EAST, kind = p.bc[side];
        if (kind == VPLBM_BC_ZEROGRAD) return {place(a, i, sj), (T)0};
        if (kind == VPLBM_BC_CONVECTIVE) return {place(a, i, sj) | EDGE_OUTLET, (T)0};
        if (kind == VPLBM_BC_VELOCITY) return {place(opp_of(a), i, j) | EDGE_ADD, wall_cu<T>(p, a, side, j)};
        if (kind != VPLBM_BC_PERIODIC) return {place(opp_of(a), i, j), (T)0};
    }
    return {place(a, si, sj), (T)0};
}

// The mailbox of a tile of w x h nodes: four values for every place around it,
// west (places 0 .. h - 1, from its rows), east (h ..), south (2 h .., from its
// columns), north (2 h + w ..): the three populations that come in there (a =
// 1, 5, 8; 3, 6, 7; 2, 5, 6; 4, 7, 8), and in the fourth, at the ends of west
// and east, the one that comes in across the corner (SW 5, SE 6, NE 7, NW 8).
// ring_item: the population of value m at place n (-1: none) and where in the
// ring it belongs.
struct RingItem {
    int a, x, y;
};
__device__ __forceinline__ RingItem ring_item(int n, int m, int w, int h)
{
    if (n < 2 * h) {
        const bool west = n < h;
        const int y = west ? n : n - h, x = west ? -1 : w;
        if (m < 3) return RingItem{west ? (m == 0 ? 1 : m == 1 ? 5 : 8) : (m == 0 ? 3 : m == 1 ? 6 : 7), x, y};
        if (y == 0) return RingItem{west ? 5 : 6, x, -1};
        if (y == h - 1) return RingItem{west ? 8 : 7, x, h};
        return RingItem{-1, 0, 0};
    }
    if (m == 3) return RingItem{-1, 0, 0};
    n -= 2 * h;
    const bool south = n < w;
    return RingItem{south ? (m == 0 ? 2 : m == 1 ? 5 : 6) : (m == 0 ? 4 : m == 1 ? 7 : 8), south ? n : n - w, south ? -1 : h};
}

// FP64 storage, MRT: a tile's sums rows [q0, q0 + qn) of step k to their
// readers.  Warp q - q0 reduces row q (a fixed order), then the first of them
// sends the reaction (q0 = 0), the last four the forces to each of their
// readers.  rows_mem: the rows, FxSum, or double where slow.  (A function of
// its own; the FP32 kernels have theirs inlined, a call cost them 8 %.)
template <typename Row>
__device__ __forceinline__ Row reduce_row(const Row *row)
{
    const int lane = threadIdx.x & 31;
    // four chains: an addition waits for the one before it in its chain only
    Row c0 = row[lane], c1 = row[32 + lane], c2 = row[64 + lane], c3 = row[96 + lane];
    for (int m = 4; m < RES_NT / 32; m += 4) {
        acc_add(c0, row[m * 32 + lane]);
        acc_add(c1, row[m * 32 + 32 + lane]);
        acc_add(c2, row[m * 32 + 64 + lane]);
        acc_add(c3, row[m * 32 + 96 + lane]);
    }
    acc_add(c0, c1);
    acc_add(c2, c3);
    acc_add(c0, c2);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc_add(c0, acc_shfl_down(c0, off));
    return c0;
}

__device__ __noinline__ void publish_sums(const ResidentLaunch &L, const void *rows_mem, double *s_tot, int i0, int j0, int q0, int qn,
                                          int k, int slot, int readers, bool slow, const BodyState *at)
{
    const int w0 = threadIdx.x >> 5, q = q0 + w0, lane = threadIdx.x & 31;
    if (w0 >= qn) return;
    if (!slow) {
        const FxSum a = reduce_row(static_cast<const FxSum *>(rows_mem) + q * RES_NT);
        if (lane == 0) s_tot[q] = q == 6 ? (double)a.lo : fx_value(a, L.p.fx.e - 59);
    } else {
        const double a = reduce_row(static_cast<const double *>(rows_mem) + q * RES_NT);
        if (lane == 0) s_tot[q] = a;
    }
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"r"(32 * qn) : "memory");
    const uint32_t tag = L.tag0 + (uint32_t)k;
    const int m = lane & 3;
    auto value = [&](int first) {   // sum first + m (the reaction has no fourth)
        double a = first == 0 && m == 3 ? 0.0 : s_tot[first + m];
        if (!slow && m == 2)        // the torque was taken about the tile's first node
            a = fma(at->q[1] - (double)j0, s_tot[first], fma((double)i0 - at->q[0], s_tot[first + 1], a));
        return make_uint2((uint32_t)__double2loint(a), (uint32_t)__double2hiint(a));
    };
    if (q0 == 0 && w0 == 0) {
        const uint2 v = value(0);
        if (lane < 4) send_pair(react_slot(L, k, slot) + 2 * m, v.x, v.y, tag);
    }
    if (q0 + qn == NPART - 1 && w0 >= qn - 4) {
        const uint2 v = value(3);
        // reader r by four lanes of warp (r >> 3) & 3 of four
        for (int r = (w0 - (qn - 4)) * 8 + (lane >> 2); r < readers; r += 32)
            send_pair(force_slot(L, k, slot, r) + 2 * m, v.x, v.y, tag);
    }
}

// Whether a solid node's pulled and own populations are in the fixed-point
// range, with a density and momentum that fx_update takes.
__device__ __forceinline__ bool fx_in_range(const FixedConsts &k, const double f[NQ], const double *own)
{
    uint32_t top = 0, low = 0xffffffffu;
    long long rho = 0, jx = 0, jy = 0;
#pragma unroll
    for (int a = 0; a < NQ; ++a) {
        const uint64_t b = fx_bits(f[a]);
        const uint32_t h = (uint32_t)(b >> 32), o = (uint32_t)(fx_bits(own[a]) >> 32);
        top = max(top, max(h, o));
        low = min(low, min(h, o));
        const long long x = fx_from(b, k.e);
        rho += x;
        jx += cx_of(a) * x;
        jy += cy_of(a) * x;
    }
    constexpr long long J = 201769274521386496LL;   // 0.35 2^59
    return top < k.hi_max && low >= k.hi_min && rho >= 1LL << 58 && rho < 3LL << 58 && jx > -J && jx < J && jy > -J && jy < J;
}

// The update of a solid node in that range (out: its place in the stage), and
// the reaction -rho a on a body of velocity bs->v that does not turn, in units
// of 2^(E - 59).
__device__ __noinline__ void fixed_solid_slow(const StepParams &p, const BodyState *bs, const double *f, double *c, long long &gx,
                                              long long &gy)
{
    double out[NQ], kept[3];
    mrt_native_f64(p, bs, true, 0.0, 0.0, f, out, kept);
    for (int a = 0; a < NQ; ++a) c[a] = out[a];
    const double s = ldexp(1.0, 59 - p.fx.e);   // |rho a| < 3: no overflow
    gx = __double2ll_rn(-kept[0] * kept[1] * s);
    gy = __double2ll_rn(-kept[0] * kept[2] * s);
}
__device__ __forceinline__ void fixed_solid(const StepParams &p, const BodyState *bs, const double f[NQ], double *c, long long &gx,
                                            long long &gy)
{
    uint64_t bits[NQ];
#pragma unroll
    for (int a = 0; a < NQ; ++a) bits[a] = fx_bits(f[a]);
    double out[NQ];
    long long rho = 0, ax = 0, ay = 0;
    if (fx_update<true>(p.fx, bits, true, fx_from_signed(fx_bits(bs->v[0])), fx_from_signed(fx_bits(bs->v[1])), out, rho, ax, ay)) {
#pragma unroll
        for (int a = 0; a < NQ; ++a) c[a] = out[a];
        const long long r8 = (long long)((uint64_t)rho << 3);
        gx = -fx_mul(r8, fx_split(2 * ax));
        gy = -fx_mul(r8, fx_split(2 * ay));
        return;
    }
    double in[NQ];
#pragma unroll
    for (int a = 0; a < NQ; ++a) in[a] = f[a];
    fixed_solid_slow(p, bs, in, c, gx, gy);
}

template <bool FIXED, typename A> struct RowT { using R = A; };
template <typename A> struct RowT<true, A> { using R = FxSum; };

// One block per SM; K nodes of 9 (FP32) or 18 (FP64) registers wait for the
// block between the pull and the update.
template <int P, int COLL, int K>
__global__ void __launch_bounds__(RES_NT, 1) vp_mrt_resident(const __grid_constant__ ResidentLaunch L)
{
    using S = typename Prec<P>::S;
    using T = typename Prec<P>::T;
    using A = typename SumT<P>::A;
    using V = typename SumT<P>::V;
    static_assert(sizeof(S) == sizeof(T), "the stage holds the arithmetic type");
    constexpr int NT = RES_NT;
    constexpr int WPV = (int)sizeof(S) / 4;   // mailbox words per value
    extern __shared__ __align__(16) unsigned char res_smem[];
    __shared__ __align__(16) BodyState s_bs[RES_TAIL_WARPS + 1];   // tiles: [step parity]; the tail: one per warp, its counters
    __shared__ int s_abort[2];   // a ring wait, the pose wait gave up
    __shared__ A s_tot[NPART - 1];   // the tile's sums
    const StepParams &p = L.p;
    const ResidentPlan &t = L.t;
    const int tid = threadIdx.x;
    if ((int)blockIdx.x == t.tiles) {
        if (!L.mute) resident_tail<P>(L, s_bs);
        return;
    }
    // solid-node sums: FP32 storage float-float, FP64 storage fixed point
    // (FIXED) or, where a solid node is out of its range, FP64
    constexpr bool FIXED = P == VPLBM_F64 && COLL == VPLBM_COLLISION_MRT;
    using R = typename RowT<FIXED, A>::R;
    R (*rows)[NT] = reinterpret_cast<R (*)[NT]>(res_smem);   // [7 sums][thread]
    A (*slow_rows)[NT] = reinterpret_cast<A (*)[NT]>(res_smem);
    S *stage = reinterpret_cast<S *>(res_smem + (NPART - 1) * NT * (P == VPLBM_F64 ? 16 : 8));
    const int pitch = (t.mw + 2) | 1;   // odd: a column of nodes is spread over the banks
    T *outlet = reinterpret_cast<T *>(stage + (size_t)pitch * (t.mh + 2) * NQ);   // [3][mh]
    // per edge node of the tile (in the order of the threads that own them):
    // its pulls [population] if it is on a lattice edge, the values it sends
    const int medge = 2 * (t.mw + t.mh);
    EdgePull<T> *epull = reinterpret_cast<EdgePull<T> *>(res_smem + L.t.edge_at);   // [9][medge]
    unsigned *post = reinterpret_cast<unsigned *>(epull + NQ * medge);               // [7][medge]: mailbox value << 4 | population
    const int nx = p.nx, ny = p.ny;
    const int tx = (int)blockIdx.x % t.ntx, ty = (int)blockIdx.x / t.ntx;
    const int i0 = tx * nx / t.ntx, j0 = ty * ny / t.nty;
    const int w = (tx + 1) * nx / t.ntx - i0, h = (ty + 1) * ny / t.nty - j0;
    const bool px = p.bc[VPLBM_WEST] == VPLBM_BC_PERIODIC, py = p.bc[VPLBM_SOUTH] == VPLBM_BC_PERIODIC;
    // neighbours (their tile columns and rows; -1: a lattice edge)
    const int cw = tx > 0 ? tx - 1 : px ? t.ntx - 1 : -1, ce = tx + 1 < t.ntx ? tx + 1 : px ? 0 : -1;
    const int rs = ty > 0 ? ty - 1 : py ? t.nty - 1 : -1, rn = ty + 1 < t.nty ? ty + 1 : py ? 0 : -1;
    const bool conv = p.bc[VPLBM_EAST] == VPLBM_BC_CONVECTIVE && i0 + w == nx;
    // a free body waits for the momentum exchanged; its sums go out within
    // the step, the others one barrier later
    const bool early = !prescribed_motion(p);

    // the state, ring included
    {
        const S *fin = static_cast<const S *>(p.fin);
        const int rw = w + 2, n = rw * (h + 2);
        for (int c = tid; c < n; c += NT) {
            const int ly = c / rw, lx = c - ly * rw;
            int i = i0 - 1 + lx, j = j0 - 1 + ly;
            if (i < 0 || i >= nx) {
                if (!px) continue;
                i = i < 0 ? i + nx : i - nx;
            }
            if (j < 0 || j >= ny) {
                if (!py) continue;
                j = j < 0 ? j + ny : j - ny;
            }
            const long long b = (long long)j * nx + i;
            S *dst = stage + (ly * pitch + lx) * NQ;
#pragma unroll
            for (int a = 0; a < NQ; ++a) dst[a] = __ldcg(fin + a * p.ps + b);   // the launch may overwrite this buffer at its end
        }
        if (conv)
            for (int q = tid; q < 3 * h; q += NT) {
                const int s = q / h, y = q - s * h;
                outlet[s * t.mh + y] = static_cast<const T *>(p.conv_in)[s * ny + j0 + y];
            }
    }
    if (tid < 2) s_abort[tid] = 0;

    // my nodes: the tile's edge first (bottom row, top row, west column, east
    // column), then the interior row by row
    unsigned node[K];
    const int edge = 2 * (w + h) - 4;   // w, h >= 3
#pragma unroll
    for (int it = 0; it < K; ++it) {
        const int n = it * NT + tid;
        int x, y;
        if (n < w) { x = n; y = 0; }
        else if (n < 2 * w) { x = n - w; y = h - 1; }
        else if (n < 2 * w + h - 2) { x = 0; y = n - 2 * w + 1; }
        else if (n < edge) { x = w - 1; y = n - 2 * w - (h - 2) + 1; }
        else { const int m = n - edge; y = m / (w - 2); x = m - y * (w - 2) + 1; ++y; }
        unsigned b = 0;
        if (n < w * h) {
            const int i = i0 + x, j = j0 + y;
            b = (unsigned)x | ((unsigned)y << 12) | ND_VALID;
            if (it == 0 && (i == 0 || i == nx - 1 || j == 0 || j == ny - 1)) {   // edge nodes are the threads' first
                b |= ND_LATTICE_EDGE;
                for (int a = 0; a < NQ; ++a) epull[a * medge + tid] = edge_pull<T>(p, a, i, j, i0, j0, pitch);
            }
            if (it == 0 && n < edge) b |= (x == 0 || x == w - 1) && (y == 0 || y == h - 1) ? ND_EDGE | ND_CORNER : ND_EDGE;
        }
        node[it] = b;
    }
    // what I receive, VPT values per 16-byte access: ring places (-1: none).
    // The tile on the other side of me receives the same from me: value m of
    // its place n is my node across from its ring place.
    constexpr int VPT = 2 / WPV;              // values per access: 2 (FP32), 1 (FP64)
    const int nunits = 2 * (w + h) * 4 / VPT;
    int rcv_at[RES_RECV][VPT];
    const uint64_t *mine = L.mail + (size_t)blockIdx.x * t.items * WPV;
    const size_t parity_stride = (size_t)t.tiles * t.items * WPV;
    for (int q = tid; q < 7 * medge; q += NT) post[q] = 0xffffffffu;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RES_RECV; ++r)
#pragma unroll
        for (int c = 0; c < VPT; ++c) {
            const int u = r * NT + tid, n = u * VPT / 4, m = (u * VPT + c) & 3;
            rcv_at[r][c] = -1;
            if (u >= nunits) continue;
            const RingItem g = ring_item(n, m, w, h);
            if (g.a < 0) continue;
            const int col = g.x < 0 ? cw : g.x == w ? ce : tx, row = g.y < 0 ? rs : g.y == h ? rn : ty;
            if (col >= 0 && row >= 0) rcv_at[r][c] = ((g.y + 1) * pitch + g.x + 1) * NQ + g.a;
            // the tile I send this value to is on the opposite side
            const int dcol = g.x < 0 ? ce : g.x == w ? cw : tx, drow = g.y < 0 ? rn : g.y == h ? rs : ty;
            if (dcol < 0 || drow < 0) continue;
            const int x = g.x < 0 ? w - 1 : g.x == w ? 0 : g.x, y = g.y < 0 ? h - 1 : g.y == h ? 0 : g.y;
            // it may be one node wider or higher across from the shared side
            const int dw = (dcol + 1) * nx / t.ntx - dcol * nx / t.ntx, dh = (drow + 1) * ny / t.nty - drow * ny / t.nty;
            const int dn = m == 3   ? (g.x < 0 ? 0 : dh) + (g.y < 0 ? 0 : dh - 1)
                           : n < h  ? n
                           : n < 2 * h ? n - h + dh
                           : n < 2 * h + w ? n - 2 * h + 2 * dh
                                       : n - 2 * h - w + 2 * dh + dw;
            // its node's place in the order of the threads; slot 0 .. 2 the
            // first side of the node, 3 .. 5 the second of a corner, 6 across
            const bool corner = (x == 0 || x == w - 1) && (y == 0 || y == h - 1);
            const int at = y == 0 ? x : y == h - 1 ? w + x : x == 0 ? 2 * w + y - 1 : 2 * w + h - 2 + y - 1;
            const int slot = m == 3 ? 6 : m + (n >= 2 * h && corner ? 3 : 0);
            post[slot * medge + at] = (unsigned)((drow * t.ntx + dcol) * t.items + dn * 4 + m) << 4 | (unsigned)g.a;
        }

    // the sums rows [q0, q0 + qn) of step k to their readers: warp q reduces
    // row q (NT / 32 adds per lane in thread order, then a shuffle tree), and
    // for a free body's forces one warp sends them all
    auto publish = [&](int q0, int qn, int k, int slot, int readers, bool slow, const BodyState *at) {
        if constexpr (FIXED) {
            publish_sums(L, res_smem, s_tot, i0, j0, q0, qn, k, slot, readers, slow, at);
            return;
        } else {
            const int q = q0 + (tid >> 5), lane = tid & 31;
            if (q >= q0 + qn) return;
            A a;
            {   // four chains: an addition waits for the one before it in its chain only
                A c[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) c[m] = rows[q][m * 32 + lane];
                for (int m = 4; m < NT / 32; m += 4)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc_add(c[e], rows[q][(m + e) * 32 + lane]);
                acc_add(c[0], c[1]);
                acc_add(c[2], c[3]);
                acc_add(c[0], c[2]);
                a = c[0];
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc_add(a, acc_shfl_down(a, off));
            const uint32_t tag = L.tag0 + (uint32_t)k;
            if (readers > 1) {   // forces, warps 0 .. 3
                if (lane == 0) s_tot[q - 3] = a;
                __syncwarp();
                asm volatile("bar.sync 1, 128;" ::: "memory");
                const uint2 v = reinterpret_cast<const uint2 *>(s_tot)[lane & 3];
                // reader r by four lanes of warp (r >> 3) & 3
                for (int r = (tid >> 5) * 8 + (lane >> 2); r < readers; r += 32)
                    send_pair(force_slot(L, k, slot, r) + 2 * (lane & 3), v.x, v.y, tag);
            } else if (lane == 0) {
                uint32_t v[2];
                memcpy(v, &a, 8);
                send_pair(q < 3 ? react_slot(L, k, slot) + 2 * q : force_slot(L, k, slot, 0) + 2 * (q - 3), v[0], v[1], tag);
                if (q == 2) send_pair(react_slot(L, k, slot) + 6, 0u, 0u, tag);   // the fourth of four
            }
        }
    };
    int owed = -1;              // the slot whose sums of the last step are still to be published
    Pair ahead{0, 0};           // words of the next pose, read early (published already on a prescribed path)
    bool own_pose = false;      // this step's pose was computed here
    bool slow = false;          // FIXED: a solid node of the tile is out of range

    for (int k = 0; k < L.nsteps; ++k) {
        const uint32_t tag = L.tag0 + (uint32_t)k;
        BodyState *bs = s_bs + (k & 1);
        __syncthreads();   // step k - 1 is in the stage
        if (owed >= 0) publish(0, early ? 3 : NPART - 1, k - 1, owed, 1, slow, s_bs + ((k - 1) & 1));
        // ---- pull of the inner nodes, which need no neighbour ----
        T f[K][NQ];
        auto pull_inner = [&](unsigned b, T g[NQ]) {
            const S *c = stage + nd_off(b, pitch);
            const S *up = c + pitch * NQ, *dn = c - pitch * NQ;
#pragma unroll
            for (int a = 0; a < NQ; ++a) g[a] = (cy_of(a) == 0 ? c : cy_of(a) > 0 ? dn : up)[a - cx_of(a) * NQ];
        };
#pragma unroll
        for (int it = 0; it < K; ++it) {
            const unsigned b = node[it];
            if ((b & ND_VALID) && !(b & ND_EDGE)) {
                pull_inner(b, f[it]);
            } else {
#pragma unroll
                for (int a = 0; a < NQ; ++a) f[it][a] = (T)0;
            }
        }
        // ---- words of this step: the ring ----
        bool ok = true;
        if (k > 0) {
            const uint64_t *box = mine + (k & 1) * parity_stride;
            unsigned pending = 0;
#pragma unroll
            for (int r = 0; r < RES_RECV; ++r)
#pragma unroll
                for (int c = 0; c < VPT; ++c) pending |= rcv_at[r][c] >= 0 ? 1u << r : 0u;
            Patience pt;
            while (pending) {
#pragma unroll
                for (int r = 0; r < RES_RECV; ++r)
                    if ((pending >> r) & 1u) {
                        const Pair v = read_pair(box + (size_t)(r * NT + tid) * 2);
                        bool here;
                        if constexpr (VPT == 2)
                            here = (rcv_at[r][0] < 0 || (uint32_t)(v.a >> 32) == tag) &&
                                   (rcv_at[r][VPT - 1] < 0 || (uint32_t)(v.b >> 32) == tag);
                        else
                            here = v.both(tag);
                        if (here) {
                            if constexpr (VPT == 2) {
                                if (rcv_at[r][0] >= 0) stage[rcv_at[r][0]] = __uint_as_float((uint32_t)v.a);
                                if (rcv_at[r][VPT - 1] >= 0) stage[rcv_at[r][VPT - 1]] = __uint_as_float((uint32_t)v.b);
                            } else {
                                reinterpret_cast<uint2 *>(stage)[rcv_at[r][0]] = make_uint2((uint32_t)v.a, (uint32_t)v.b);
                            }
                            pending &= ~(1u << r);
                        }
                    }
                if (pending && pt.out(L.timeout_ns)) {
                    atomicOr(p.err, ERR_TIMEOUT);
                    ok = false;
                    break;
                }
            }
        }
        if (!ok) s_abort[0] = 1;
        __syncthreads();
        if (s_abort[0]) return;   // uniform

        // ---- pull of the edge nodes ----
        if (node[0] & ND_EDGE) {
            const unsigned b = node[0];
            if (!(b & ND_LATTICE_EDGE)) {
                pull_inner(b, f[0]);
            } else {
#pragma unroll
                for (int a = 0; a < NQ; ++a) {
                    const EdgePull<T> e = epull[a * medge + tid];
                    T v = stage[e.at & 0xffffffu];
                    if (e.at & EDGE_ADD) v = fma((T)(6.0 * w_of(a)) * par<T>(p.rho0, p.rho0f), e.cu, v);
                    if (cx_of(a) < 0) {
                        T *prev = outlet + outlet_slot(a) * t.mh + nd_y(b);
                        if (e.at & EDGE_OUTLET) v = par<T>(p.conv_k1, p.conv_k1f) * *prev + par<T>(p.conv_k2, p.conv_k2f) * v;
                        if (conv && i0 + nd_x(b) == nx - 1) *prev = v;   // the outlet's record of this step
                    }
                    f[0][a] = v;
                }
            }
        }
        // the pose: a free body's comes last, and only the update needs it; a
        // tile that met the body has it already
        const int mine_of_pose = tid - (NT - POSE_WORDS / 2);   // two words
        if (mine_of_pose >= 0 && !own_pose) {
            if (!wait_pair(L, pose_slot(L, k) + 2 * mine_of_pose, tag, ahead)) s_abort[1] = 1;
            reinterpret_cast<uint2 *>(bs)[mine_of_pose] = make_uint2((uint32_t)ahead.a, (uint32_t)ahead.b);
        }
        __syncthreads();
        if (s_abort[1]) return;
        const int4 range = make_int4(bs->ilo, bs->ihi, bs->jlo, bs->jhi);
        const int4 rect = make_int4((int)bs->pad0, (int)(bs->pad0 >> 32), bs->pad[0], bs->pad[1]);
        const bool sums = tx >= rect.x && tx < rect.x + rect.z && ty >= rect.y && ty < rect.y + rect.w;
        const bool near = sums && range.x <= range.y;

        // ---- update ----
        const bool send = k + 1 < L.nsteps;
        if (send && !early && mine_of_pose >= 0) ahead = read_pair(pose_slot(L, k + 1) + 2 * mine_of_pose);
        // my edge node's values to the neighbours, as soon as it is updated
        auto post_edge = [&]() {
            const unsigned b = node[0];
            if (!send || !(b & ND_EDGE)) return;
            const S *c = stage + nd_off(b, pitch);
            uint64_t *out = L.mail + ((k + 1) & 1) * parity_stride;
            // the three values of a side (mailbox neighbours) and one across a corner
            auto side = [&](int m0) {
                const unsigned e = post[m0 * medge + tid], e1 = post[(m0 + 1) * medge + tid], e2 = post[(m0 + 2) * medge + tid];
                if (e == 0xffffffffu) return;
                uint64_t *dst = out + (size_t)(e >> 4) * WPV;
                if constexpr (WPV == 1) {
                    const uint32_t *v = reinterpret_cast<const uint32_t *>(c);
                    send_pair(dst, v[e & 15u], v[e1 & 15u], tag + 1);
                    send_word(dst + 2, v[e2 & 15u], tag + 1);
                } else {
                    const uint2 *v = reinterpret_cast<const uint2 *>(c);
                    const uint2 v0 = v[e & 15u], v1 = v[e1 & 15u], v2 = v[e2 & 15u];
                    send_pair(dst, v0.x, v0.y, tag + 1);
                    send_pair(dst + 2, v1.x, v1.y, tag + 1);
                    send_pair(dst + 4, v2.x, v2.y, tag + 1);
                }
            };
            side(0);
            if (b & ND_CORNER) {
                side(3);
                const unsigned e = post[6 * medge + tid];
                if (e == 0xffffffffu) return;
                uint64_t *dst = out + (size_t)(e >> 4) * WPV;
                if constexpr (WPV == 1) {
                    send_word(dst, reinterpret_cast<const uint32_t *>(c)[e & 15u], tag + 1);
                } else {
                    const uint2 v = reinterpret_cast<const uint2 *>(c)[e & 15u];
                    send_pair(dst, v.x, v.y, tag + 1);
                }
            }
        };
        const int slot = (ty - rect.y) * rect.z + tx - rect.x;
        if (sums && !near && tid < 8)   // no solid node anywhere
            send_pair((tid < 4 ? force_slot(L, k, 0, 0) : react_slot(L, k, 0)) + 2 * (tid & 3), 0u, 0u, tag);
        auto lever = [&](unsigned b, T &dx, T &dy) {
            if constexpr (P == VPLBM_F64) {
                dx = (double)(i0 + nd_x(b)) - bs->q[0];
                dy = (double)(j0 + nd_y(b)) - bs->q[1];
            } else {
                dx = (float)(i0 + nd_x(b) - bs->xi) - bs->xf;
                dy = (float)(j0 + nd_y(b) - bs->yi) - bs->yf;
            }
        };
        unsigned solid = 0;   // my solid nodes
        if (near) {
            // the momentum exchanged by a solid node: pulled minus own, before
            // the own populations are overwritten
            A ex_[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc_zero(ex_[q]);
            auto exchange = [&](unsigned b, const T g[NQ], T dx, T dy) {
                const S *c = stage + nd_off(b, pitch);
                V ex = 0, ey = 0;
#pragma unroll
                for (int a = 1; a < NQ; ++a) {
                    const V d = (V)g[a] - (V)c[a];
                    ex += cx_of(a) * d;
                    ey += cy_of(a) * d;
                }
                acc_add(ex_[0], ex);
                acc_add(ex_[1], ey);
                acc_add(ex_[2], (V)dx * ey - (V)dy * ex);
                acc_add(ex_[3], (V)1);
            };
            bool bad = false;
#pragma unroll
            for (int it = 0; it < K; ++it) {
                const unsigned b = node[it];
                const int i = i0 + nd_x(b), j = j0 + nd_y(b);
                if (!(b & ND_VALID) || i < range.x || i > range.y || j < range.z || j > range.w) continue;
                T dxl = 0, dyl = 0;
                if (!body_chi<P, SHAPE_ANY>(p.body, p.r2f, bs, i, j, dxl, dyl)) continue;
                solid |= 1u << it;
                if constexpr (FIXED) bad = bad || !fx_in_range(p.fx, f[it], stage + nd_off(b, pitch));
                else exchange(b, f[it], dxl, dyl);
            }
            if constexpr (FIXED) {
                // a body that turns, or moves fast, takes the FP64 code too
                const uint64_t v0 = fx_bits(bs->v[0]), v1 = fx_bits(bs->v[1]);
                bad = bad || !p.fx.ok || p.fx.forced || bs->v[2] != 0.0 || ((v0 >> 32) & 0x7fffffffu) >= 0x3fd00000u ||
                      ((v1 >> 32) & 0x7fffffffu) >= 0x3fd00000u;
                slow = __syncthreads_or(bad);
            }
            if constexpr (FIXED) {
                if (!slow) {
                    FxSum sum[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc_zero(sum[q]);
#pragma unroll
                    for (int it = 0; it < K; ++it) {
                        if (!((solid >> it) & 1u)) continue;
                        const unsigned b = node[it];
                        const S *c = stage + nd_off(b, pitch);
                        long long ex = 0, ey = 0;
#pragma unroll
                        for (int a = 1; a < NQ; ++a) {
                            const long long g = fx_from(fx_bits(f[it][a]), p.fx.e) - fx_from(fx_bits(c[a]), p.fx.e);
                            if (cx_of(a)) ex += cx_of(a) > 0 ? g : -g;
                            if (cy_of(a)) ey += cy_of(a) > 0 ? g : -g;
                        }
                        acc_add(sum[0], fx_term(ex));
                        acc_add(sum[1], fx_term(ey));
                        acc_add(sum[2], fx_term(ey, nd_x(b)));
                        acc_add(sum[2], fx_term(ex, -nd_y(b)));
                        sum[3].lo += 1;
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) rows[3 + q][tid] = sum[q];
                } else {
#pragma unroll
                    for (int it = 0; it < K; ++it) {
                        if (!((solid >> it) & 1u)) continue;
                        T dx, dy;
                        lever(node[it], dx, dy);
                        exchange(node[it], f[it], dx, dy);
                    }
                }
            }
            if (!FIXED || slow) {
#pragma unroll
                for (int q = 0; q < 4; ++q) slow_rows[3 + q][tid] = ex_[q];
            }
            if (early) {
                __syncthreads();
                publish(3, 4, k, slot, 1 + rect.z * rect.w, slow, bs);
            }
        }
        // the penalization's reaction, summed over my solid nodes
        A part[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) acc_zero(part[q]);
        auto react = [&](T dx, T dy, T rho, T ax, T ay) {
            const V fx = -(V)rho * (V)ax, fy = -(V)rho * (V)ay;
            acc_add(part[0], fx);
            acc_add(part[1], fy);
            acc_add(part[2], (V)dx * fy - (V)dy * fx);
        };
        FxSum fpart[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) acc_zero(fpart[q]);
        constexpr bool PAIRS = P == VPLBM_F32_DEV && COLL == VPLBM_COLLISION_MRT;
        if constexpr (PAIRS) {
            // two of my nodes at a time on paired lanes
#pragma unroll
            for (int it = 0; it + 1 < K; it += 2) {
                const unsigned b0 = node[it], b1 = node[it + 1];
                const bool pen = near && __any_sync(0xffffffffu, (solid >> it) & 3u);
                const bool first = (b0 & ND_VALID) != 0, second = (b1 & ND_VALID) != 0;
                if (!__any_sync(0xffffffffu, first)) continue;
                float2 f2[NQ];
#pragma unroll
                for (int a = 0; a < NQ; ++a) f2[a] = make_float2(f[it][a], f[it + 1][a]);
                S *c0 = stage + nd_off(b0, pitch), *c1 = stage + nd_off(b1, pitch);
                auto store = [&](int a, float2 v) {
                    if (first) c0[a] = v.x;
                    if (second) c1[a] = v.y;
                };
                if (pen) {
                    const bool s0 = (solid >> it) & 1u, s1 = (solid >> it) & 2u;
                    float2 dx, dy, ax, ay;
                    lever(b0, dx.x, dy.x);
                    lever(b1, dx.y, dy.y);
                    const float2 rho = mrt_dev_pair_chi(p, f2, s0, s1, dx, dy, bs, store, ax, ay);
                    if (s0) react(dx.x, dy.x, rho.x, ax.x, ay.x);
                    if (s1) react(dx.y, dy.y, rho.y, ax.y, ay.y);
                } else {
                    float ax, ay;
                    mrt_dev_lanes<Lane2>(p, f2, false, 0.f, 0.f, bs, store, ax, ay);
                }
                if (it == 0) post_edge();
            }
        }
        // the rest (all of them for FP64 storage and BGK) one at a time
#pragma unroll
        for (int it = PAIRS ? K / 2 * 2 : 0; it < K; ++it) {
            const unsigned b = node[it];
            auto update_one = [&]() {
                S *c = stage + nd_off(b, pitch);
                T dxl = 0, dyl = 0, cr = 0, cax = 0, cay = 0;
                const bool chi = (solid >> it) & 1u;
                if constexpr (FIXED) {
                    if (chi && !slow) {
                        long long gx = 0, gy = 0;
                        fixed_solid(p, bs, f[it], c, gx, gy);   // -rho a
                        acc_add(fpart[0], fx_term(gx));
                        acc_add(fpart[1], fx_term(gy));
                        acc_add(fpart[2], fx_term(gy, nd_x(b)));
                        acc_add(fpart[2], fx_term(gx, -nd_y(b)));
                        return;
                    }
                }
                if (chi) lever(b, dxl, dyl);
                node_collide_to<P, COLL>(p, bs, chi, dxl, dyl, f[it], [&](int a, T v) { c[a] = v; }, cr, cax, cay);
                if (chi) react(dxl, dyl, cr, cax, cay);
            };
            if (b & ND_VALID) update_one();
            if (it == 0) post_edge();
        }
        if (near) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if constexpr (FIXED) {
                    if (!slow) rows[q][tid] = fpart[q];
                    else slow_rows[q][tid] = part[q];
                } else {
                    rows[q][tid] = part[q];
                }
            }
        }
        owed = near ? slot : -1;
        own_pose = early && near && send;
        if (own_pose && tid >= NT - 32 && !tile_next_pose<A>(L, k, s_bs, slot)) s_abort[1] = 1;
    }
    if (owed >= 0) {
        __syncthreads();
        publish(0, early ? 3 : NPART - 1, L.nsteps - 1, owed, 1, slow, s_bs + ((L.nsteps - 1) & 1));
    }

    // the state after the last step (every thread its own nodes)
    S *fout = static_cast<S *>(L.fout);
#pragma unroll
    for (int it = 0; it < K; ++it) {
        const unsigned b = node[it];
        if (!(b & ND_VALID)) continue;
        const S *c = stage + nd_off(b, pitch);
        S *dst = fout + (long long)(j0 + nd_y(b)) * nx + i0 + nd_x(b);
#pragma unroll
        for (int a = 0; a < NQ; ++a) dst[a * p.ps] = c[a];
    }
    if (conv) {
        __syncthreads();
        for (int q = tid; q < 3 * h; q += NT) {
            const int s = q / h, y = q - s * h;
            static_cast<T *>(L.conv_out)[s * ny + j0 + y] = outlet[s * t.mh + y];
        }
    }
}

template <int P, int COLL, int K>
cudaError_t launch_k(const ResidentLaunch &L, cudaStream_t stream)
{
    cudaError_t e = cudaFuncSetAttribute(vp_mrt_resident<P, COLL, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, L.t.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.t.tiles + 1);
    cfg.blockDim = dim3(RES_NT);
    cfg.dynamicSmemBytes = L.t.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, vp_mrt_resident<P, COLL, K>, L);
}

template <int P, int COLL> cudaError_t launch_pc(const ResidentLaunch &L, cudaStream_t stream)
{
    if (L.t.k == 1) return launch_k<P, COLL, 1>(L, stream);
    if (L.t.k == 2) return launch_k<P, COLL, 2>(L, stream);
    if constexpr (P == VPLBM_F32_DEV) {
        if (L.t.k == 3) return launch_k<P, COLL, 3>(L, stream);
        if (L.t.k == 4) return launch_k<P, COLL, 4>(L, stream);
        if (L.t.k == 5) return launch_k<P, COLL, 5>(L, stream);
        // six too: a kernel of its own would be 3 to 5 % faster there (1100 x
        // 400: 5.59 against 5.85 us a step) and is one more to build
        if (L.t.k <= 7) return launch_k<P, COLL, 7>(L, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// Nodes per thread for tiles of w x h nodes (0: not possible), where the edge
// tables start in the dynamic shared memory, and its size.
int resident_k(int precision, int w, int h, int *edge_at, int *smem)
{
    const int maxk = precision == VPLBM_F32_DEV ? 7 : precision == VPLBM_F64 ? 2 : 0;
    const long long es = precision == VPLBM_F64 ? 8 : 4;
    for (int k = 1; k <= maxk; ++k) {
        if ((long long)w * h > (long long)k * RES_NT) continue;
        // the sums' rows, the stage, the outlet record; then the edge tables
        const long long at = ((NPART - 1) * (long long)RES_NT * 2 * es + (NQ * ((w + 2LL) | 1) * (h + 2LL) + 3LL * h) * es + 15) / 16 * 16;
        const long long bytes = at + 2LL * (w + h) * (NQ * 2 * es + 7 * 4);
        if (bytes > 225 * 1024 || (precision == VPLBM_F64 ? 8 : 4) * (w + h) > RES_RECV * RES_NT || 2 * (w + h) > RES_NT || w < 3 ||
            h < 3 || w > 4095 || h > 4095)
            return 0;
        *edge_at = (int)at;
        *smem = (int)bytes;
        return k;
    }
    return 0;
}

size_t resident_bytes(const ResidentPlan &t, int precision, size_t *poses, size_t *parts)
{
    const size_t mail = (size_t)2 * t.tiles * t.items * (precision == VPLBM_F64 ? 2 : 1) * sizeof(uint64_t);
    *poses = (mail + 255) / 256 * 256;
    *parts = *poses + (size_t)t.pose_ring * POSE_WORDS * sizeof(uint64_t);
    return *parts + (size_t)RES_PART_RING * (t.part_copies + 1) * t.part_slots * 8 * sizeof(uint64_t);
}

// P11, P12 / m, P21, P22 / m of advance_free.
void resident_rk(const DevBody &b, double rk[3][4])
{
    for (int d = 0; d < 3; ++d) {
        const double a = d < 2 ? b.inv_mass : b.inv_inertia, k = b.stiff[d] * a, c = b.damp[d] * a;
        // powers of L = [[0, 1], [-k, -c]]
        const double l2[4] = {-k, -c, k * c, c * c - k};
        const double l3[4] = {l2[2], l2[3], -k * l2[0] - c * l2[2], -k * l2[1] - c * l2[3]};
        rk[d][0] = 1.0 + l2[0] / 6.0 + l3[0] / 24.0;
        rk[d][1] = (0.5 + l2[1] / 6.0 + l3[1] / 24.0) * a;
        rk[d][2] = -0.5 * k + l2[2] / 6.0 + l3[2] / 24.0;
        rk[d][3] = (1.0 - 0.5 * c + l2[3] / 6.0 + l3[3] / 24.0) * a;
    }
}

cudaError_t launch_resident(int precision, const ResidentLaunch &L, cudaStream_t stream)
{
    const bool bgk = L.p.collision == VPLBM_COLLISION_BGK;
    switch (precision) {
    case VPLBM_F32_DEV:
        return bgk ? launch_pc<VPLBM_F32_DEV, VPLBM_COLLISION_BGK>(L, stream)
                   : launch_pc<VPLBM_F32_DEV, VPLBM_COLLISION_MRT>(L, stream);
    case VPLBM_F64:
        return bgk ? launch_pc<VPLBM_F64, VPLBM_COLLISION_BGK>(L, stream)
                   : launch_pc<VPLBM_F64, VPLBM_COLLISION_MRT>(L, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace vplbm
