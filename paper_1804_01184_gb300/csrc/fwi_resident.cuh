// fwi_resident.cuh -- time-step kernels that keep the wavefield on chip (sm_103a).
//
// A launch advances some shots by many steps.  Each shot's grid is cut into tx x tz tiles, one
// CTA a tile, all CTAs of the launch resident at once (cooperative launch).  Global memory sees
// only what the caller asked for (pressure history, traces, final state) and the tiles'
// boundary exchange.
//
// Layout.  A warp owns R rows of its tile, a lane one float4 of columns of each: lane l holds
// column group l - 1 (4 columns), so lanes 1 .. ng are the tile's own groups (at most 30) and
// lanes 0 and ng + 1 the groups beside it.  The cells' fields and model sit in registers for the
// whole launch.  The x-stencil of p reads shared rows, that of v_x shuffles within the warp, and
// the z-stencils read the rows of other warps from shared memory.  The tile's rows are
// extended by the M rows above and M - 1 below whose v_z the divergence of its own rows reads.
//
// One exchange a step: the halo's velocities are updated here too (the neighbours compute the
// same values from the same operands), so only pressure crosses tiles, 2M - 1 cells deep.
// Neighbours send each value as an 8-byte word (step tag, float) into the receiver's mailbox
// in global memory (L2); the receiver polls the words themselves, so a step waits for one
// store-to-load latency, without flags or fences.  Two mailbox slots alternate: a CTA sends
// step n + 2 only after it has the neighbour's step n + 1, which the neighbour computed after
// reading step n.
//
// Every cell's arithmetic is the streaming kernels' (fwi_warp.cuh), operation for operation, so
// results are bitwise theirs for every tiling.
#pragma once
#include "fwi_warp.cuh"

namespace fwi {

constexpr int RES_RC = 64;      // receivers of a tile listed in shared memory
// a wait gives up after this many polls unless told otherwise (a poll is an L2 round trip, ~1 us: a
// few seconds)
constexpr int RES_POLLS = 1 << 21;
enum : int { ST_ETIMEOUT = 16 };

// How long a launch's waits last, and where an expired one is recorded besides the operation's status
// word (the engine's word in host memory, or null).
struct ResWait {
    int polls;
    int *expired;
};

// A wait of this block has expired.
__device__ __forceinline__ void res_expired(const ResWait &w, int *status, int *abort)
{
    *reinterpret_cast<volatile int *>(abort) = 1;
    atomicOr(status, ST_ETIMEOUT);
    if (w.expired) *reinterpret_cast<volatile int *>(w.expired) = 1;
}

// Shape of a resident CTA: up to NW warps of R rows of 30 column groups.
template <int M_, int R_, int NW_>
struct ResShape {
    static constexpr int M = M_, R = R_, NW = NW_;
    static constexpr int HR = 2 * M - 1;             // depth of the pressure halo
    static constexpr int G = 30, W = 4 * G;          // own column groups, columns
    static constexpr int E = NW * R, H = E - HR;     // extended rows (from -M on), own rows
    static constexpr int PP = W + 16;                // pitch of a p row: column c at c + 8
    static constexpr int PZ = 128;                   // pitch of a v_z row: lane l at 4 l
};

// Rows a warp, against 12 warps of 168 registers an SM (24 of fields and model a row).  Three leave
// the windows in registers and give short tiles all 12 warps; four (five at 4th order, whose
// windows are shorter) make taller tiles, for grids that would not fit and for the engine,
// whose launches other jobs fill.  Measured (us a step, 8th order): 10 shots of 201^2 2.9 with three
// rows, 3.2 with four; 16 warps of two 3.4 (their tiles need two launches); 8 warps of eight 4.3.
using ResFwd2 = ResShape<2, 5, 12>;
using ResFwd2s = ResShape<2, 3, 12>;
using ResFwd4 = ResShape<4, 4, 12>;
using ResFwd4s = ResShape<4, 3, 12>;

// Cut of a shot's grid: tx x tz tiles; the first grem (hrem) tiles have one column group (row)
// more than gbase (hbase).
struct ResCut {
    int tx, tz, gbase, grem, hbase, hrem;
};

// A tile's mailbox, in words: two slots of 2M - 1 rows from above and below and 8 columns from the
// left and right, and a ring of 4 for the lower right diagonal tile's first cell (diagonal
// tiles do not wait on each other).  The engine's are sized for the cut's largest tile (half
// a job's fields hold state while it runs); a single call's for the shape's, whose constants
// save 2 to 5 % of a step.
template <class S, bool FIT>
struct ResMail {
    int w, below, left, right, slot, all;    // pitch of a row; offsets in a slot; words of a slot, of a tile
    __host__ __device__ explicit ResMail(const ResCut &c)
    {
        w = 4 * (c.gbase + (c.grem > 0));
        const int h = c.hbase + (c.hrem > 0);
        below = S::HR * w;
        left = 2 * below;
        right = left + 8 * h;
        slot = right + 8 * h;
        all = 2 * slot + 4;
    }
};

template <class S>
struct ResMail<S, false> {
    static constexpr int w = S::W, below = S::HR * w, left = 2 * below, right = left + 8 * S::H, slot = right + 8 * S::H,
                         all = 2 * slot + 4;
    __host__ __device__ explicit ResMail(const ResCut &) {}
};

// The stencil's weights (negated: -c_k dt / dx) in both halves of a pair, as the packed
// multiply-adds read them.
struct ResStencil {
    float2 nc[4];
};

__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    float2 r;
    asm("{\n\t.reg .b64 a, b, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tsub.rn.f32x2 r, a, b;\n\t"
        "mov.b64 {%0, %1}, r;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
// c + s (a - b), both halves of s equal: ptap
__device__ __forceinline__ float4 rtap(const float2 &s, const float4 &a, const float4 &b, const float4 &c)
{
    return cat4(__ffma2_rn(s, sub2(lo2(a), lo2(b)), lo2(c)), __ffma2_rn(s, sub2(hi2(a), hi2(b)), hi2(c)));
}
__device__ __forceinline__ float4 rscale(const float2 &s, const float4 &b)
{
    return cat4(__fmul2_rn(s, lo2(b)), __fmul2_rn(s, hi2(b)));
}
// row_dplus / row_dminus of a float4 b with the float4 a to its left and c to its right
template <int M, bool PLUS>
__device__ __forceinline__ float4 row_diff(const float4 &a, const float4 &b, const float4 &c, const float2 *cf)
{
    const float w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    float o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float g = 0.f;
#pragma unroll
        for (int k = 1; k <= M; ++k)
            g = PLUS ? fmaf(cf[k - 1].x, w[4 + q + k] - w[4 + q - k + 1], g) : fmaf(cf[k - 1].x, w[4 + q + k - 1] - w[4 + q - k], g);
        o[q] = g;
    }
    return make_float4(o[0], o[1], o[2], o[3]);
}

struct ResFwdArgs {
    const float *p0, *vx0, *vz0;    // state before step n0 of shot 0 (null: zero)
    float *p1, *vx1, *vz1;          // state after step n1 - 1 (null: not written); may be the
                                    // state before (every step exchanges: a neighbour has read it)
    float *hist;                    // p^{n0} .. p^{n1}, one slot a step (null: not kept)
    long long slot;                 // floats between history slots
    Model mo;
    Dims d;
    ResStencil st;
    Source src;
    const long long *ridx;          // receivers (traces non-null)
    const float *rw;
    float *traces;                  // [shots][nr][nt]
    int nr, nt;
    int n0, n1;
    ResCut cut;
    ResWait wait;
    unsigned long long *mail;       // [shots][tiles] mailboxes (ResMail), cleared before the launch
};

// Four values and their step tag as two 16-byte stores; each 8-byte word is written whole.
__device__ __forceinline__ void mail_put4(unsigned long long *m, const float4 &v, unsigned tag)
{
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(m), "l"(t | __float_as_uint(v.x)),
                 "l"(t | __float_as_uint(v.y))
                 : "memory");
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(m + 2), "l"(t | __float_as_uint(v.z)),
                 "l"(t | __float_as_uint(v.w))
                 : "memory");
}

// What a launch works on: a single call's arguments (CAP 1), or the engine's table, whose job j
// takes blocks start[j] .. start[j + 1) (tiles within shots).
constexpr int RES_CAP = 24;
template <class A, int CAP>
struct ResBatch {
    int njobs;
    int start[CAP + 1];
    A jobs[CAP];
};

template <class A>
struct ResBatch<A, 1> {
    A job;
};

template <class A>
__device__ __forceinline__ const A &res_job(const ResBatch<A, 1> &t, int &block)
{
    block = blockIdx.x;
    return t.job;
}

template <class A, int CAP>
__device__ __forceinline__ const A &res_job(const ResBatch<A, CAP> &t, int &block)
{
    int j = 0;
    block = blockIdx.x;
    while (j + 1 < t.njobs && t.start[j + 1] <= block) ++j;
    block -= t.start[j];
    return t.jobs[j];
}

struct MailWord4 {
    unsigned long long w[4];
};

__device__ __forceinline__ void mail_get4(const unsigned long long *m, MailWord4 &r)
{
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(r.w[0]), "=l"(r.w[1]) : "l"(m) : "memory");
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(r.w[2]), "=l"(r.w[3]) : "l"(m + 2) : "memory");
}

__device__ __forceinline__ bool mail_ready(const MailWord4 &r, unsigned tag)
{
    return (unsigned)(r.w[0] >> 32) == tag && (unsigned)(r.w[1] >> 32) == tag && (unsigned)(r.w[2] >> 32) == tag &&
           (unsigned)(r.w[3] >> 32) == tag;
}

__device__ __forceinline__ float4 mail_value(const MailWord4 &r)
{
    return make_float4(__uint_as_float((unsigned)r.w[0]), __uint_as_float((unsigned)r.w[1]),
                       __uint_as_float((unsigned)r.w[2]), __uint_as_float((unsigned)r.w[3]));
}

// The mailboxes that a tile may touch, for the checked builds: its shot's.
struct MailSpan {
#ifdef FWI_CHECKED
    const unsigned long long *base;
    long long words;
    int *status;
    __device__ MailSpan(const unsigned long long *b, long long w, int *s) : base(b), words(w), status(s) {}
    __device__ __forceinline__ bool has(const unsigned long long *m, int len) const { return in_field(m - base, len, words, status); }
#else
    __device__ MailSpan(const unsigned long long *, long long, int *) {}
    __device__ __forceinline__ bool has(const unsigned long long *, int) const { return true; }
#endif
};

// This CTA's tile.
struct ResTile {
    int t, s;            // tile of its shot, shot of the launch
    int g0, ng;          // first column group, groups
    int z0, h;           // first row, rows
    bool L, R, U, D;     // has a neighbour
};

__device__ __forceinline__ ResTile res_tile(const ResCut &c, int block)
{
    ResTile T;
    const int n = c.tx * c.tz;
    T.s = block / n;
    T.t = block - T.s * n;
    const int tj = T.t / c.tx, ti = T.t - tj * c.tx;
    T.g0 = ti * c.gbase + min(ti, c.grem);
    T.ng = c.gbase + (ti < c.grem);
    T.z0 = tj * c.hbase + min(tj, c.hrem);
    T.h = c.hbase + (tj < c.hrem);
    T.L = ti > 0;
    T.R = ti + 1 < c.tx;
    T.U = tj > 0;
    T.D = tj + 1 < c.tz;
    return T;
}

// Receivers of a tile (those whose first corner cell is its own).
struct ResRec {
    int n;               // receivers of the tile (above RES_RC every step scans them all)
    int diag;            // a receiver reads the cell past the tile's lower right corner
    int r[RES_RC], off[RES_RC];
    float w[RES_RC][4];
};

// Shared memory of a forward CTA.
template <class S>
struct __align__(16) ResFwdSmem {
    float p[S::E + S::HR][S::PP];            // row e at [e + HR]
    float vz[S::E + 2 * S::M][S::PZ];        // row e at [e + 2M]
    float2 az[S::E], azh[S::E];              // row e at [e + M], in both halves
    int sj[4], si[4];                        // the shot's source cells relative to the tile
    float sw[4];
    ResRec rec;
    int abort;                               // a wait of this CTA expired
};

// The tile's receivers (order irrelevant: each writes its own trace); offsets for pitch PP.
// lim: floats from own cell (0, 0) to the end of the field (checked builds)
__device__ __forceinline__ void res_receivers(ResRec &rc, const ResTile &T, const Dims &d, const long long *ridx,
                                              const float *rw, int nr, int PP, int tid, int lim, int *stt)
{
    for (int k = tid; k < nr; k += blockDim.x) {
        const long long o = ridx[4 * k];
        const int j = (int)(o / d.Px) - T.z0, i = (int)(o % d.Px) - 4 * T.g0;
        if (!FWI_IN(j >= 0 && j < T.h && i >= 0 && i < 4 * T.ng, j * PP + i, PP + 2, lim, stt)) continue;
        if (j == T.h - 1 && i == 4 * T.ng - 1) rc.diag = 1;
        const int e = atomicAdd(&rc.n, 1);
        if (e >= RES_RC) continue;
        rc.r[e] = k;
        rc.off[e] = j * PP + i;
        for (int c = 0; c < 4; ++c) rc.w[e][c] = rw[4 * k + c];
    }
}

// trace[s][r][n] of the tile's receivers from p^{n+1} (own cells and halo); `p`: own cell (0, 0), lim as above
__device__ __forceinline__ void res_sample(const ResRec &rc, const ResTile &T, const Dims &d, const long long *ridx,
                                           const float *rw, float *traces, int nr, int nt, int n, const float *p, int PP,
                                           int tid, int lim, int *stt)
{
    if (rc.n <= RES_RC) {
        for (int k = tid; k < rc.n; k += blockDim.x) {
            const float *q = p + rc.off[k];
            float v = 0.f;
            v = fmaf(rc.w[k][0], q[0], v);
            v = fmaf(rc.w[k][1], q[1], v);
            v = fmaf(rc.w[k][2], q[PP], v);
            v = fmaf(rc.w[k][3], q[PP + 1], v);
            traces[((long long)T.s * nr + rc.r[k]) * nt + n] = v;
        }
        return;
    }
    for (int k = tid; k < nr; k += blockDim.x) {
        const long long o = ridx[4 * k];
        const int j = (int)(o / d.Px) - T.z0, i = (int)(o % d.Px) - 4 * T.g0;
        if (!FWI_IN(j >= 0 && j < T.h && i >= 0 && i < 4 * T.ng, j * PP + i, PP + 2, lim, stt)) continue;
        const float *q = p + j * PP + i;
        float v = 0.f;
        v = fmaf(rw[4 * k], q[0], v);
        v = fmaf(rw[4 * k + 1], q[1], v);
        v = fmaf(rw[4 * k + 2], q[PP], v);
        v = fmaf(rw[4 * k + 3], q[PP + 1], v);
        traces[((long long)T.s * nr + k) * nt + n] = v;
    }
}

// What a thread receives: the float4 tid, tid + nt, ... of the halo; the first two kept as
// (mailbox word, offset from the field's own cell (0, 0)).
template <class S, class Mail>
struct ResRecv {
    int n, w0, o0, w1, o1;
    __device__ ResRecv(const ResTile &T, const Mail &B, int tid, int nt)
    {
        n = (T.U + T.D) * S::HR * T.ng + 2 * (T.L + T.R) * T.h;
        item(T, B, tid, w0, o0);
        item(T, B, tid + nt, w1, o1);
    }
    __device__ __forceinline__ void item(const ResTile &T, const Mail &B, int k, int &word, int &off) const
    {
        const int nrow = S::HR * T.ng, nU = T.U ? nrow : 0, nD = T.D ? nrow : 0, nL = T.L ? 2 * T.h : 0;
        if (k >= n) k = 0;
        if (k < nU + nD) {
            const bool up = k < nU;
            const int q = up ? k : k - nU, r = q / T.ng, g = 4 * (q - r * T.ng);
            word = (up ? 0 : B.below) + r * B.w + g;
            off = ((up ? -S::HR : T.h) + r) * S::PP + g;
        } else {
            k -= nU + nD;
            const bool left = k < nL;
            if (!left) k -= nL;
            word = (left ? B.left : B.right) + 4 * k;
            off = (k >> 1) * S::PP + (left ? -8 : 4 * T.ng) + 4 * (k & 1);
        }
    }
    // words of step `tag` of this tile's mailbox slot m into the halo of the field whose own cell
    // (0, 0) is at p; false when a wait expired (a limit of 0 expires wherever the tile has neighbours)
    __device__ __forceinline__ bool get(const unsigned long long *m, const ResTile &T, const Mail &B, float *p,
                                        unsigned tag, int tid, int nt, int polls, const MailSpan &box) const
    {
        int spin = 0;
        if (tid < n && box.has(m + w0, 4)) {
            const bool two = tid + nt < n && box.has(m + w1, 4);
            MailWord4 a, b;
            mail_get4(m + w0, a);
            if (two) mail_get4(m + w1, b);
            while (!mail_ready(a, tag) && ++spin < polls) mail_get4(m + w0, a);
            st4(p + o0, mail_value(a));
            if (two) {
                while (!mail_ready(b, tag) && ++spin < polls) mail_get4(m + w1, b);
                st4(p + o1, mail_value(b));
            }
            for (int k = tid + 2 * nt; k < n; k += nt) {
                int w, o;
                item(T, B, k, w, o);
                if (!box.has(m + w, 4)) continue;
                mail_get4(m + w, a);
                while (!mail_ready(a, tag) && ++spin < polls) mail_get4(m + w, a);
                st4(p + o, mail_value(a));
            }
        }
        return spin < polls || n == 0;
    }
};

// What a lane sends of its own rows: up and down (rows within HR of the edge), and left or right
// (the two groups at the edge; tiles with such a neighbour have at least 4 groups).
template <class S, class Mail>
struct ResSend {
    unsigned long long *ud, *lr;         // word of row 0 in the neighbour's slot; null: none
    int dn;                              // down's offset from up
    bool up, down;                       // this warp has rows for the neighbour
    __device__ ResSend(unsigned long long *box, const ResTile &T, const ResCut &c, const Mail &B, int g, int e0)
    {
        const bool own = g >= 0 && g < T.ng;
        up = own && T.U && e0 < S::HR && e0 + S::R > 0;
        down = own && T.D && e0 + S::R > T.h - S::HR && e0 < T.h;
        ud = box - (long long)c.tx * B.all + B.below + 4 * g;
        dn = 2 * c.tx * B.all - B.below - (T.h - S::HR) * B.w;
        lr = own && T.L && g < 2 ? box - B.all + B.right + 4 * g
             : own && T.R && g >= T.ng - 2 ? box + B.all + B.left + 4 * (g - (T.ng - 2)) : nullptr;
    }
    __device__ __forceinline__ void put(const ResTile &T, const Mail &B, int slot, int e0, const float4 (&v)[S::R], unsigned tag,
                                        const MailSpan &shot) const
    {
        constexpr int R = S::R;
        if (lr)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (e0 + r >= 0 && e0 + r < T.h && shot.has(lr + slot + (e0 + r) * 8, 4)) mail_put4(lr + slot + (e0 + r) * 8, v[r], tag);
        if (up)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (e0 + r >= 0 && e0 + r < S::HR && shot.has(ud + slot + (e0 + r) * B.w, 4))
                    mail_put4(ud + slot + (e0 + r) * B.w, v[r], tag);
        if (down)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (e0 + r >= T.h - S::HR && e0 + r < T.h && shot.has(ud + dn + slot + (e0 + r) * B.w, 4))
                    mail_put4(ud + dn + slot + (e0 + r) * B.w, v[r], tag);
    }
};

// The neighbours' float4 of a row held across the warp, those components an order-2M D- reads
template <int M>
__device__ __forceinline__ void warp_sides(const float4 &b, float4 &l, float4 &r)
{
    const unsigned all = 0xffffffffu;
    l = r = f4(0.f);
    if (M > 3) l.x = __shfl_up_sync(all, b.x, 1);
    if (M > 2) l.y = __shfl_up_sync(all, b.y, 1);
    l.z = __shfl_up_sync(all, b.z, 1);
    l.w = __shfl_up_sync(all, b.w, 1);
    r.x = __shfl_down_sync(all, b.x, 1);
    if (M > 2) r.y = __shfl_down_sync(all, b.y, 1);
    if (M > 3) r.z = __shfl_down_sync(all, b.z, 1);
}

// Forward steps n0 .. n1 - 1.
template <class S, int CAP>
__global__ void __launch_bounds__(32 * S::NW, 1) k_res_fwd(const __grid_constant__ ResBatch<ResFwdArgs, CAP> t)
{
    constexpr int M = S::M, R = S::R, HR = S::HR, PP = S::PP, PZ = S::PZ;
    extern __shared__ __align__(16) unsigned char fwi_smem[];
    ResFwdSmem<S> &sh = *reinterpret_cast<ResFwdSmem<S> *>(fwi_smem);
    int block;
    const ResFwdArgs &a = res_job(t, block);
    const ResCut &c = a.cut;
    const Dims &d = a.d;
    const Model &mo = a.mo;
    const int tid = threadIdx.x, lane = tid & 31, nt = blockDim.x;
    const ResTile T = res_tile(c, block);
    const long long so = (long long)T.s * d.Np;
    int *stt = mo.status;

    for (int k = tid; k < (int)(sizeof(ResFwdSmem<S>) / 4); k += nt) reinterpret_cast<int *>(fwi_smem)[k] = 0;
    __syncthreads();
    for (int k = tid; k < S::E; k += nt) {
        const int j = T.z0 - M + k;
        if (j >= 0 && j < d.Nz) {
            sh.az[k] = make_float2(mo.az[j], mo.az[j]);
            sh.azh[k] = make_float2(mo.azh[j], mo.azh[j]);
        }
    }
    if (tid < 4) {
        const long long o = a.src.idx[4 * T.s + tid];
        sh.sj[tid] = (int)(o / d.Px) - T.z0;
        sh.si[tid] = (int)(o % d.Px) - 4 * T.g0;
        sh.sw[tid] = a.src.w[4 * T.s + tid];
    }
    if (a.traces) res_receivers(sh.rec, T, d, a.ridx, a.rw, a.nr, PP, tid, S::E * PP - 8, stt);
    float *const p00 = &sh.p[HR][8];                      // own cell (0, 0)
    if (a.p0)   // initial pressure of the tile and its halo
        for (int k = tid; k < (T.h + 2 * HR) * (T.ng + 4); k += nt) {
            const int row = k / (T.ng + 4) - HR, g = k % (T.ng + 4) - 2;
            const int j = T.z0 + row, i = 4 * (T.g0 + g);
            const bool rin = row >= 0 && row < T.h, gin = g >= 0 && g < T.ng;
            if (!rin && !gin) continue;                   // corners no stencil reads
            if (FWI_IN(j >= 0 && j < d.Nz && i >= 0 && i < d.Nx, j * d.Px + i, 4, d.Np, stt))
                st4(p00 + row * PP + 4 * g, ld4(a.p0 + so + j * d.Px + i));
        }
    __syncthreads();

    // this lane's cells: group g, extended rows e0 .. e0 + R - 1
    const int g = lane - 1, e0 = (tid >> 5) * R - M, col = 4 * (T.g0 + g);
    const bool own = g >= 0 && g < T.ng, side = (g == -1 || g == T.ng) && col >= 0 && col < d.Nx;
    const int go = (T.z0 + e0) * d.Px + col;
    const float4 axv = ldg_if(mo.ax + col, own), axhv = ldg_if(mo.axh + col, own || side);
    float4 p[R], vx[R], vz[R], Kv[R], bx[R], bz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = e0 + r, j = T.z0 + e, o = go + r * d.Px;
        const bool grid = j >= 0 && j < d.Nz, rin = e >= 0 && e < T.h, zin = e < T.h + M - 1;
        const bool fx = FWI_IN(grid && rin && (own || side), o, 4, d.Np, stt), fz = FWI_IN(grid && zin && own, o, 4, d.Np, stt);
        Kv[r] = ldg_if(mo.K + o, fz && rin);
        bx[r] = ldg_if(mo.bx + o, fx);
        bz[r] = ldg_if(mo.bz + o, fz);
        p[r] = vx[r] = vz[r] = f4(0.f);
        if (a.p0) {
            if (fx) vx[r] = ld4(a.vx0 + so + o);
            if (fz) vz[r] = ld4(a.vz0 + so + o);
            p[r] = ld4(p00 + e * PP + 4 * g);   // own cells and halo; zero elsewhere
        }
        if (a.hist && fz && rin) st4(a.hist + so + o, p[r]);
    }
    bool hsrc = false;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        hsrc |= own && sh.si[k] >= 4 * g && sh.si[k] < 4 * g + 4 && sh.sj[k] >= max(e0, 0) && sh.sj[k] < min(e0 + R, T.h);
    using Mail = ResMail<S, (CAP > 1)>;
    const Mail mb(c);
    unsigned long long *const box = a.mail + ((long long)T.s * c.tx * c.tz + T.t) * mb.all;
    const MailSpan shot(box - (long long)T.t * mb.all, (long long)c.tx * c.tz * mb.all, stt), mine(box, mb.all, stt);
    const ResSend<S, Mail> send(box, T, c, mb, g, e0);
    const ResRecv<S, Mail> recv(T, mb, tid, nt);
    float *const prow = p00 + e0 * PP + 4 * g;            // p of (e0, g)
    float *const zrow = &sh.vz[e0 + 2 * M][4 * lane];     // v_z of (e0, g)
    const float2 *const azr = sh.az + e0 + M, *const azhr = sh.azh + e0 + M;
    float *hrow = a.hist ? a.hist + so + go : nullptr;
    const float2 *const nc = a.st.nc;
#ifdef FWI_CHECKED
    bool sound = FWI_SPAN(sh.p, prow - (M - 1) * PP - 4, prow + (R - 1 + M) * PP + 8, stt) &&
                 FWI_SPAN(sh.vz, zrow - M * PZ, zrow + (R + M - 2) * PZ + 4, stt) && in_field(e0 + M, R, S::E, stt);
    for (int k = tid; k < recv.n; k += nt) {
        int w, o;
        recv.item(T, mb, k, w, o);
        sound = FWI_SPAN(sh.p, p00 + o, p00 + o + 4, stt) && sound;
    }
    if (__syncthreads_or(!sound)) return;   // (the neighbours' waits for this tile expire)
#endif

    const bool inner = e0 >= 0 && e0 + R <= T.h;          // every row of the warp is an own row
    float wn = hsrc ? __ldg(a.src.wav + a.n0) : 0.f;
    for (int n = a.n0; n < a.n1; ++n) {
        // ---------------------------------------------------------------- velocities
        {
            float4 w[R + HR];   // p rows e0 - M + 1 .. e0 + R - 1 + M
#pragma unroll
            for (int q = 0; q < M - 1; ++q) w[q] = ld4(prow + (q - (M - 1)) * PP);
#pragma unroll
            for (int q = 0; q < R; ++q) w[M - 1 + q] = p[q];
#pragma unroll
            for (int q = 0; q < M; ++q) w[M - 1 + R + q] = ld4(prow + (R + q) * PP);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float4 gz = f4(0.f);
#pragma unroll
                for (int k = 1; k <= M; ++k) gz = rtap(nc[k - 1], w[r + M - 1 + k], w[r + M - k], gz);
                vz[r] = pmul(rscale(azhr[r], axv), pfma(bz[r], gz, vz[r]));
                st4(zrow + r * PZ, vz[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 gx = row_diff<M, true>(ld4(prow + r * PP - 4), p[r], ld4(prow + r * PP + 4), nc);
            vx[r] = pmul(rscale(azr[r], axhv), pfma(bx[r], gx, vx[r]));
        }
        __syncthreads();
        // ------------------------------------------------------------------ pressure
        const unsigned tag = (unsigned)(n - a.n0) + 1u;
        const int slot = (n & 1) * mb.slot;
        if (hrow) hrow += a.slot;
        {
            float4 w[R + HR];   // v_z rows e0 - M .. e0 + R - 1 + M - 1
#pragma unroll
            for (int q = 0; q < M; ++q) w[q] = ld4(zrow + (q - M) * PZ);
#pragma unroll
            for (int q = 0; q < R; ++q) w[M + q] = vz[q];
#pragma unroll
            for (int q = 0; q < M - 1; ++q) w[M + R + q] = ld4(zrow + (R + q) * PZ);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float4 l, q;
                warp_sides<M>(vx[r], l, q);
                float4 dv = row_diff<M, false>(l, vx[r], q, nc);
#pragma unroll
                for (int k = 1; k <= M; ++k) dv = rtap(nc[k - 1], w[r + M + k - 1], w[r + M - k], dv);
                p[r] = pmul(rscale(azr[r], axv), pfma(Kv[r], dv, p[r]));
            }
            if (hsrc)
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int e = e0 + r, i = sh.si[k] - 4 * g;
                        if (sh.sj[k] == e && e >= 0 && e < T.h && i >= 0 && i < 4)
                            add_source<false>(p[r], i, __fmul_rn(comp(Kv[r], i), wn), sh.sw[k]);
                    }
            send.put(T, mb, slot, e0, p, tag, shot);
            if (own) {
                if (inner) {
#pragma unroll
                    for (int r = 0; r < R; ++r) st4(prow + r * PP, p[r]);
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        if (e0 + r >= 0 && e0 + r < T.h) st4(prow + r * PP, p[r]);
                }
                if (hrow)
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        if (e0 + r >= 0 && e0 + r < T.h && FWI_IN(true, (long long)go + r * d.Px, 4, d.Np, stt))
                            st4(hrow + r * d.Px, p[r]);
            }
            if (hsrc && n + 1 < a.n1) wn = __ldg(a.src.wav + n + 1);
        }
        // ------------------------------------------------------------------ exchange
        if (e0 <= 0 && e0 + R > 0 && g == 0 && T.U && T.L) {   // the first cell, for the upper left diagonal tile
            float v = 0.f;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (e0 + r == 0) v = p[r].x;
            unsigned long long *const dg = box - (long long)(c.tx + 1) * mb.all + 2 * mb.slot + (n & 3);
            if (shot.has(dg, 1))
                asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(dg), "l"((unsigned long long)tag << 32 | __float_as_uint(v))
                             : "memory");
        }
        bool ok = recv.get(box + slot, T, mb, p00, tag, tid, nt, a.wait.polls, mine);
        if (tid == 0 && sh.rec.diag && T.R && T.D && mine.has(box + 2 * mb.slot + (n & 3), 1)) {
            unsigned long long v = 0;
            int spin = 0;
            do {
                asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(box + 2 * mb.slot + (n & 3)) : "memory");
            } while ((unsigned)(v >> 32) != tag && ++spin < a.wait.polls);
            ok = ok && spin < a.wait.polls;
            p00[T.h * PP + 4 * T.ng] = __uint_as_float((unsigned)v);
        }
        if (!ok) res_expired(a.wait, stt, &sh.abort);
        __syncthreads();
        if (*reinterpret_cast<volatile int *>(&sh.abort)) break;
        if (a.traces) res_sample(sh.rec, T, d, a.ridx, a.rw, a.traces, a.nr, a.nt, n, p00, PP, tid, S::E * PP - 8, stt);
        // the halo's pressure: the groups beside the tile, and the rows above and below it
        if (!own || !inner)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (!own || e0 + r < 0 || e0 + r >= T.h) p[r] = ld4(prow + r * PP);
    }
    if (a.vx1)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = e0 + r, o = go + r * d.Px;
            if (FWI_IN(own && e >= 0 && e < T.h, o, 4, d.Np, stt)) {
                if (a.p1) st4(a.p1 + so + o, p[r]);
                st4(a.vx1 + so + o, vx[r]);
                st4(a.vz1 + so + o, vz[r]);
            }
        }
}

// ------------------------------------------------------------- adjoint steps (S7)
//
// Reverse steps nhi, nhi - 1, .. nlo of the adjoint scheme (see fwi_warp.cuh) with the gradient
// products, kept on chip like the forward steps.  The exchanged field is q = K d_p pbar, which is
// all the stencils read of pbar beyond a tile.  The accumulators and the step's forward pressure
// (copied in one step ahead by cp.async) sit in shared memory.  The receivers' residual of the
// next step is added to pbar, with its K-gradient term, before q is formed; the caller has added
// step nhi's.

constexpr int RES_ENT = 256;    // injection cells of a tile listed in shared memory
// three rows: 4.8 us a step for 10 shots of 201^2, four 6.0 (the second window spills)
using ResAdj2 = ResShape<2, 4, 12>;
using ResAdj2s = ResShape<2, 3, 12>;
using ResAdj4 = ResShape<4, 4, 12>;
using ResAdj4s = ResShape<4, 3, 12>;

struct ResAdjArgs {
    const float *ap0, *avx0, *avz0;   // pbar^{nhi+1} (injected), vbar of the launch's shots
    float *ap1, *avx1, *avz1;         // pbar^{nlo}, vbar after step nlo; other buffers, or with two
                                      // steps or more (one exchange) the same
    const float *pn;                  // p^{nlo}, one slot a step
    long long slot;
    float *accK, *accBx, *accBz;      // FP32 accumulators, read and written once
    Model mo;
    Dims d;
    ResStencil st;                    // c_k dt / dx (not negated)
    const long long *ridx;
    const float *rw;
    const int *rl;                    // chains of footprint entries that share a cell
    const float *res;                 // [shots][nr][nt]
    int nr, nt;
    int nhi, nlo;
    ResCut cut;
    ResWait wait;
    unsigned long long *mail;
};

template <class S>
struct __align__(16) ResAdjSmem {
    float q[S::E + S::HR][S::PP];            // row e at [e + HR], column c at [c + 8]
    float pn[2][S::E + S::HR][S::PP];        // forward pressure of this step and the next
    float bz[S::E + 2 * S::M][S::PZ];        // b_z u_z: row e at [e + 2M]
    float acc[3][S::E][128];                 // K, b_x, b_z: row e at [e + M], lane l at 4 l
    float inj[S::E][128];                    // the next step's injection, zero off the receivers
    float2 az[S::E], azh[S::E];              // row e at [e + M], in both halves
    int cell[RES_ENT], ent[RES_ENT];         // injection cells: offset in inj, first footprint entry
    int has[S::E];                           // the row holds an injection cell
    int nent;
    int abort;
};

// acc + v as the streaming kernels' red.global.add.f32 adds it: subnormals flush to zero
__device__ __forceinline__ float4 add_ftz(const float4 &a, const float4 &v)
{
    float4 r;
    asm("add.rn.ftz.f32 %0, %1, %2;" : "=f"(r.x) : "f"(a.x), "f"(v.x));
    asm("add.rn.ftz.f32 %0, %1, %2;" : "=f"(r.y) : "f"(a.y), "f"(v.y));
    asm("add.rn.ftz.f32 %0, %1, %2;" : "=f"(r.z) : "f"(a.z), "f"(v.z));
    asm("add.rn.ftz.f32 %0, %1, %2;" : "=f"(r.w) : "f"(a.w), "f"(v.w));
    return r;
}

template <class S, int CAP>
__global__ void __launch_bounds__(32 * S::NW, 1) k_res_adj(const __grid_constant__ ResBatch<ResAdjArgs, CAP> t)
{
    constexpr int M = S::M, R = S::R, HR = S::HR, PP = S::PP, PZ = S::PZ;
    extern __shared__ __align__(16) unsigned char fwi_smem[];
    ResAdjSmem<S> &sh = *reinterpret_cast<ResAdjSmem<S> *>(fwi_smem);
    int block;
    const ResAdjArgs &a = res_job(t, block);
    const ResCut &c = a.cut;
    const Dims &d = a.d;
    const Model &mo = a.mo;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
    const ResTile T = res_tile(c, block);
    const long long so = (long long)T.s * d.Np;
    int *stt = mo.status;

    for (int k = tid; k < (int)(sizeof(ResAdjSmem<S>) / 4); k += nt) reinterpret_cast<int *>(fwi_smem)[k] = 0;
    __syncthreads();
    for (int k = tid; k < S::E; k += nt) {
        const int j = T.z0 - M + k;
        if (j >= 0 && j < d.Nz) {
            sh.az[k] = make_float2(mo.az[j], mo.az[j]);
            sh.azh[k] = make_float2(mo.azh[j], mo.azh[j]);
        }
    }
    // the cell of footprint entry k in inj, -1 when another entry leads its chain or it is not here
    auto entry_cell = [&](int k) {
        if (!(a.rl[k] & CHAIN_FIRST)) return -1;
        const long long o = a.ridx[k];
        const int j = (int)(o / d.Px) - T.z0, i = (int)(o % d.Px) - 4 * T.g0;
        const int at = (j + M) * 128 + 4 + i;
        return FWI_IN(j >= 0 && j < T.h && i >= 0 && i < 4 * T.ng, at, 1, S::E * 128, stt) ? at : -1;
    };
    for (int k = tid; k < 4 * a.nr; k += nt) {
        const int o = entry_cell(k);
        if (o < 0) continue;
        sh.has[o >> 7] = 1;
        const int e = atomicAdd(&sh.nent, 1);
        if (e < RES_ENT) {
            sh.cell[e] = o;
            sh.ent[e] = k;
        }
    }
    float *const q00 = &sh.q[HR][8], *const p00 = &sh.pn[0][HR][8];   // own cell (0, 0)
    constexpr int PB = (S::E + HR) * PP;                              // floats of a pn buffer
    // q of the tile and its halo
    for (int k = tid; k < (T.h + 2 * HR) * (T.ng + 4); k += nt) {
        const int row = k / (T.ng + 4) - HR, g = k % (T.ng + 4) - 2;
        const int j = T.z0 + row, i = 4 * (T.g0 + g), o = j * d.Px + i;
        const bool rin = row >= 0 && row < T.h, gin = g >= 0 && g < T.ng;
        if (!rin && !gin) continue;                   // corners no stencil reads
        if (FWI_IN(j >= 0 && j < d.Nz && i >= 0 && i < d.Nx, o, 4, d.Np, stt))
            st4(q00 + row * PP + 4 * g, pmul(pmul(mo.az[j], ldg4(mo.ax + i)), pmul(ldg4(mo.K + o), ld4(a.ap0 + so + o))));
    }
    // forward pressure of step n: rows -(M - 1) .. h + M - 1, the tile's groups and one beside each
    auto fetch = [&](int n, int buf) {
        const float *src = a.pn + (long long)(n - a.nlo) * a.slot + so;
        const int gl = lane - 1, i = 4 * (T.g0 + gl);
        const bool ok = gl <= T.ng && i >= 0 && i < d.Nx;
        for (int row = warp - (M - 1); row < T.h + M; row += nw) {
            const int j = T.z0 + row;
            if (FWI_IN(ok && j >= 0 && j < d.Nz, j * d.Px + i, 4, d.Np, stt))
                cp16(p00 + buf * PB + row * PP + 4 * gl, src, j * d.Px + i, true);
        }
        cp_commit();
    };
    fetch(a.nhi, 0);

    // this lane's cells: group g, extended rows e0 .. e0 + R - 1
    const int g = lane - 1, e0 = warp * R - M, col = 4 * (T.g0 + g);
    const bool own = g >= 0 && g < T.ng, side = (g == -1 || g == T.ng) && col >= 0 && col < d.Nx;
    const int go = (T.z0 + e0) * d.Px + col;
    const float4 axv = ldg_if(mo.ax + col, own), axhv = ldg_if(mo.axh + col, own || side);
    float4 pb[R], ux[R], uz[R], Kv[R], bx[R], bz[R];
    float *const acck = &sh.acc[0][e0 + M][4 * lane], *const accx = &sh.acc[1][e0 + M][4 * lane],
                *const accz = &sh.acc[2][e0 + M][4 * lane];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = e0 + r, j = T.z0 + e, o = go + r * d.Px;
        const bool grid = j >= 0 && j < d.Nz, rin = e >= 0 && e < T.h, zin = e < T.h + M - 1;
        const bool fx = FWI_IN(grid && rin && (own || side), o, 4, d.Np, stt), fz = FWI_IN(grid && zin && own, o, 4, d.Np, stt);
        Kv[r] = ldg_if(mo.K + o, fz && rin);
        bx[r] = ldg_if(mo.bx + o, fx);
        bz[r] = ldg_if(mo.bz + o, fz);
        pb[r] = ux[r] = uz[r] = f4(0.f);
        if (fx) ux[r] = ld4(a.avx0 + so + o);
        if (fz) uz[r] = ld4(a.avz0 + so + o);
        if (fz && rin) {
            pb[r] = ld4(a.ap0 + so + o);
            st4(acck + r * 128, ld4(a.accK + so + o));
            st4(accx + r * 128, ld4(a.accBx + so + o));
            st4(accz + r * 128, ld4(a.accBz + so + o));
        }
    }
    __syncthreads();
    unsigned hinj = 0;                                    // this warp's rows with injection cells
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (own && sh.has[e0 + r + M]) hinj |= 1u << r;
    using Mail = ResMail<S, (CAP > 1)>;
    const Mail mb(c);
    unsigned long long *const box = a.mail + ((long long)T.s * c.tx * c.tz + T.t) * mb.all;
    const MailSpan shot(box - (long long)T.t * mb.all, (long long)c.tx * c.tz * mb.all, stt), mine(box, mb.all, stt);
    const ResSend<S, Mail> send(box, T, c, mb, g, e0);
    const ResRecv<S, Mail> recv(T, mb, tid, nt);
    float *const qrow = q00 + e0 * PP + 4 * g;
    const float *const prow = p00 + e0 * PP + 4 * g;
    float *const zrow = &sh.bz[e0 + 2 * M][4 * lane];
    const float2 *const azr = sh.az + e0 + M, *const azhr = sh.azh + e0 + M;
    const float2 *const cf = a.st.nc;
#ifdef FWI_CHECKED
    bool sound = FWI_SPAN(sh.q, qrow - (M - 1) * PP - 4, qrow + (R - 1 + M) * PP + 8, stt) &&
                 FWI_SPAN(sh.pn[0], prow - (M - 1) * PP - 4, prow + (R - 1 + M) * PP + 8, stt) &&
                 FWI_SPAN(sh.bz, zrow - M * PZ, zrow + (R + M - 2) * PZ + 4, stt) && in_field(e0 + M, R, S::E, stt) &&
                 in_field(T.h + M - 1 + HR, 1, S::E + HR, stt);   // the last row of pressure fetched
    for (int k = tid; k < recv.n; k += nt) {
        int w, o;
        recv.item(T, mb, k, w, o);
        sound = FWI_SPAN(sh.q, q00 + o, q00 + o + 4, stt) && sound;
    }
    cp_wait<0>();
    if (__syncthreads_or(!sound)) return;   // (the neighbours' waits for this tile expire)
#endif
    const bool inner = e0 >= 0 && e0 + R <= T.h;
    const float *const rs = a.res + (long long)T.s * a.nr * a.nt;
    const int n4 = 4 * a.nr, nent = sh.nent;
    // this thread's first listed cell: its leading residual, loaded a step ahead
    const bool lead = nent <= RES_ENT && tid < nent;
    const int ek = lead ? sh.ent[tid] : 0, eo = lead ? sh.cell[tid] : 0;
    float rv = lead && a.nhi > a.nlo ? rs[(long long)(ek >> 2) * a.nt + a.nhi - 1] : 0.f;
    // sum over the chain of entry k of its residuals at step n, the leading one given
    auto chain = [&](int k, int n, float first) {
        float v = __fmul_rn(a.rw[k], first);
        for (int m = a.rl[k] & (CHAIN_FIRST - 1); m < n4; m = a.rl[m] & (CHAIN_FIRST - 1))
            v = fmaf(a.rw[m], rs[(long long)(m >> 2) * a.nt + n], v);
        return v;
    };
    cp_wait<0>();
    __syncthreads();

    for (int n = a.nhi; n >= a.nlo; --n) {
        const int it = a.nhi - n, buf = it & 1;
        const float *const pr = prow + buf * PB;
        if (n > a.nlo) fetch(n - 1, buf ^ 1);
        else cp_commit();
        // the injection of step n - 1 (added below, after pbar^n)
        if (n > a.nlo) {
            if (nent <= RES_ENT) {
                if (lead) {
                    (&sh.inj[0][0])[eo] = chain(ek, n - 1, rv);
                    if (n - 1 > a.nlo) rv = rs[(long long)(ek >> 2) * a.nt + n - 2];
                }
                for (int k = tid + nt; k < nent; k += nt) {
                    const int e = sh.ent[k];
                    (&sh.inj[0][0])[sh.cell[k]] = chain(e, n - 1, rs[(long long)(e >> 2) * a.nt + n - 1]);
                }
            } else {
                for (int k = tid; k < n4; k += nt) {
                    const int o = entry_cell(k);
                    if (o >= 0) (&sh.inj[0][0])[o] = chain(k, n - 1, rs[(long long)(k >> 2) * a.nt + n - 1]);
                }
            }
        }
        // ---------------------------------------------------------------- velocities
        {
            float4 w[R + HR];   // q rows e0 - M + 1 .. e0 + R - 1 + M
#pragma unroll
            for (int k = 0; k < R + HR; ++k) w[k] = ld4(qrow + (k - (M - 1)) * PP);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float4 gq = f4(0.f);
#pragma unroll
                for (int k = 1; k <= M; ++k) gq = rtap(cf[k - 1], w[r + M - 1 + k], w[r + M - k], gq);
                uz[r] = pmul(rscale(azhr[r], axv), padd(uz[r], gq));
                st4(zrow + r * PZ, pmul(bz[r], uz[r]));
                const float4 gx = row_diff<M, true>(ld4(qrow + r * PP - 4), w[r + M - 1], ld4(qrow + r * PP + 4), cf);
                ux[r] = pmul(rscale(azr[r], axhv), padd(ux[r], gx));
            }
        }
        {
            float4 w[R + HR];   // p^n rows
#pragma unroll
            for (int k = 0; k < R + HR; ++k) w[k] = ld4(pr + (k - (M - 1)) * PP);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float4 gp = f4(0.f);
#pragma unroll
                for (int k = 1; k <= M; ++k) gp = rtap(cf[k - 1], w[r + M - 1 + k], w[r + M - k], gp);
                st4(accz + r * 128, add_ftz(ld4(accz + r * 128), pmul(uz[r], gp)));
                const float4 gx = row_diff<M, true>(ld4(pr + r * PP - 4), w[r + M - 1], ld4(pr + r * PP + 4), cf);
                st4(accx + r * 128, add_ftz(ld4(accx + r * 128), pmul(ux[r], gx)));
            }
        }
        __syncthreads();
        // ------------------------------------------------------------------ pressure
        const unsigned tag = (unsigned)it + 1u;
        const int slot = (it & 1) * mb.slot;
        {
            float4 w[R + HR];   // b_z u_z rows e0 - M .. e0 + R - 1 + M - 1
#pragma unroll
            for (int k = 0; k < M; ++k) w[k] = ld4(zrow + (k - M) * PZ);
#pragma unroll
            for (int k = 0; k < R; ++k) w[M + k] = pmul(bz[k], uz[k]);
#pragma unroll
            for (int k = 0; k < M - 1; ++k) w[M + R + k] = ld4(zrow + (R + k) * PZ);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 bu = pmul(bx[r], ux[r]);
                float4 l, rr;
                warp_sides<M>(bu, l, rr);
                float4 dv = row_diff<M, false>(l, bu, rr, cf);
#pragma unroll
                for (int k = 1; k <= M; ++k) dv = rtap(cf[k - 1], w[r + M + k - 1], w[r + M - k], dv);
                pb[r] = pfma(rscale(azr[r], axv), pb[r], dv);
                st4(acck + r * 128, add_ftz(ld4(acck + r * 128), pmul(ld4(pr + r * PP), dv)));
            }
        }
        if (n == a.nlo) break;
        if (hinj) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (hinj >> r & 1) {
                    const float4 v = ld4(&sh.inj[e0 + r + M][4 * lane]), p = ld4(pr + r * PP);
                    float4 k = ld4(acck + r * 128);
                    if (v.x != 0.f) { pb[r].x = __fadd_rn(pb[r].x, v.x); k.x = fmaf(v.x, p.x, k.x); }
                    if (v.y != 0.f) { pb[r].y = __fadd_rn(pb[r].y, v.y); k.y = fmaf(v.y, p.y, k.y); }
                    if (v.z != 0.f) { pb[r].z = __fadd_rn(pb[r].z, v.z); k.z = fmaf(v.z, p.z, k.z); }
                    if (v.w != 0.f) { pb[r].w = __fadd_rn(pb[r].w, v.w); k.w = fmaf(v.w, p.w, k.w); }
                    st4(acck + r * 128, k);
                }
        }
        // ------------------------------------------------------------------ exchange
        {
            float4 q[R];
#pragma unroll
            for (int r = 0; r < R; ++r) q[r] = pmul(rscale(azr[r], axv), pmul(Kv[r], pb[r]));
            send.put(T, mb, slot, e0, q, tag, shot);
            if (own)
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (inner || (e0 + r >= 0 && e0 + r < T.h)) st4(qrow + r * PP, q[r]);
        }
        if (!recv.get(box + slot, T, mb, q00, tag, tid, nt, a.wait.polls, mine)) res_expired(a.wait, stt, &sh.abort);
        cp_wait<0>();
        __syncthreads();
        if (*reinterpret_cast<volatile int *>(&sh.abort)) break;
    }
    cp_wait<0>();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = e0 + r, o = go + r * d.Px;
        if (FWI_IN(own && e >= 0 && e < T.h, o, 4, d.Np, stt)) {
            st4(a.ap1 + so + o, pb[r]);
            st4(a.avx1 + so + o, ux[r]);
            st4(a.avz1 + so + o, uz[r]);
            st4(a.accK + so + o, ld4(acck + r * 128));
            st4(a.accBx + so + o, ld4(accx + r * 128));
            st4(a.accBz + so + o, ld4(accz + r * 128));
        }
    }
}

// ------------------------------------------------------------------------ Born steps (S6)
//
// Background and scattered wavefields (see k_born_warp) stepped together on chip: the forward
// kernel's structure with two of everything.  Three rows a warp; the model's perturbation sits in
// shared memory, read by its own lane alone.  10 shots of 201^2: 6.6 us a step (two rows 7.6).
using ResBorn2 = ResShape<2, 3, 12>;
using ResBorn4 = ResShape<4, 3, 12>;

struct ResBornArgs {
    const float *p0, *vx0, *vz0, *q0, *ux0, *uz0;   // state before step n0 of shot 0 (null p0: zero)
    float *p1, *vx1, *vz1, *q1, *ux1, *uz1;         // state after step n1 - 1 (null p1: not written); may
                                                    // be the state before
    Model mo;
    Pert pe;
    Dims d;
    ResStencil st;
    Source src;
    const long long *ridx;
    const float *rw;
    float *traces;                                  // [shots][nr][nt], samples of q (null: none)
    int nr, nt;
    int n0, n1;
    ResCut cut;
    ResWait wait;
    unsigned long long *mail, *mailq;               // p's and q's mailboxes
};

template <class S>
struct __align__(16) ResBornSmem {
    float p[S::E + S::HR][S::PP], q[S::E + S::HR][S::PP];            // row e at [e + HR]
    float vz[S::E + 2 * S::M][S::PZ], uz[S::E + 2 * S::M][S::PZ];    // row e at [e + 2M]
    float dm[3][S::E][128];                  // dK, dbx, dbz: row e at [e + M], lane l at 4 l
    float2 az[S::E], azh[S::E];
    int sj[4], si[4];
    float sw[4];
    ResRec rec;
    int abort;
};

template <class S, int CAP>
__global__ void __launch_bounds__(32 * S::NW, 1) k_res_born(const __grid_constant__ ResBatch<ResBornArgs, CAP> t)
{
    constexpr int M = S::M, R = S::R, HR = S::HR, PP = S::PP, PZ = S::PZ;
    extern __shared__ __align__(16) unsigned char fwi_smem[];
    ResBornSmem<S> &sh = *reinterpret_cast<ResBornSmem<S> *>(fwi_smem);
    int block;
    const ResBornArgs &a = res_job(t, block);
    const ResCut &c = a.cut;
    const Dims &d = a.d;
    const Model &mo = a.mo;
    const int tid = threadIdx.x, lane = tid & 31, nt = blockDim.x;
    const ResTile T = res_tile(c, block);
    const long long so = (long long)T.s * d.Np;
    int *stt = mo.status;

    for (int k = tid; k < (int)(sizeof(ResBornSmem<S>) / 4); k += nt) reinterpret_cast<int *>(fwi_smem)[k] = 0;
    __syncthreads();
    for (int k = tid; k < S::E; k += nt) {
        const int j = T.z0 - M + k;
        if (j >= 0 && j < d.Nz) {
            sh.az[k] = make_float2(mo.az[j], mo.az[j]);
            sh.azh[k] = make_float2(mo.azh[j], mo.azh[j]);
        }
    }
    if (tid < 4) {
        const long long o = a.src.idx[4 * T.s + tid];
        sh.sj[tid] = (int)(o / d.Px) - T.z0;
        sh.si[tid] = (int)(o % d.Px) - 4 * T.g0;
        sh.sw[tid] = a.src.w[4 * T.s + tid];
    }
    if (a.traces) res_receivers(sh.rec, T, d, a.ridx, a.rw, a.nr, PP, tid, S::E * PP - 8, stt);
    float *const p00 = &sh.p[HR][8], *const q00 = &sh.q[HR][8];
    if (a.p0)   // initial fields of the tile and its halo
        for (int k = tid; k < (T.h + 2 * HR) * (T.ng + 4); k += nt) {
            const int row = k / (T.ng + 4) - HR, g = k % (T.ng + 4) - 2;
            const int j = T.z0 + row, i = 4 * (T.g0 + g);
            const bool rin = row >= 0 && row < T.h, gin = g >= 0 && g < T.ng;
            if (!rin && !gin) continue;
            if (FWI_IN(j >= 0 && j < d.Nz && i >= 0 && i < d.Nx, j * d.Px + i, 4, d.Np, stt)) {
                st4(p00 + row * PP + 4 * g, ld4(a.p0 + so + j * d.Px + i));
                st4(q00 + row * PP + 4 * g, ld4(a.q0 + so + j * d.Px + i));
            }
        }
    __syncthreads();

    const int g = lane - 1, e0 = (tid >> 5) * R - M, col = 4 * (T.g0 + g);
    const bool own = g >= 0 && g < T.ng, side = (g == -1 || g == T.ng) && col >= 0 && col < d.Nx;
    const int go = (T.z0 + e0) * d.Px + col;
    const float4 axv = ldg_if(mo.ax + col, own), axhv = ldg_if(mo.axh + col, own || side);
    float4 p[R], vx[R], vz[R], q[R], ux[R], uz[R], Kv[R], bx[R], bz[R];
    float *const dk = &sh.dm[0][e0 + M][4 * lane], *const dbx = &sh.dm[1][e0 + M][4 * lane], *const dbz = &sh.dm[2][e0 + M][4 * lane];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = e0 + r, j = T.z0 + e, o = go + r * d.Px;
        const bool grid = j >= 0 && j < d.Nz, rin = e >= 0 && e < T.h, zin = e < T.h + M - 1;
        const bool fx = FWI_IN(grid && rin && (own || side), o, 4, d.Np, stt), fz = FWI_IN(grid && zin && own, o, 4, d.Np, stt);
        Kv[r] = ldg_if(mo.K + o, fz && rin);
        bx[r] = ldg_if(mo.bx + o, fx);
        bz[r] = ldg_if(mo.bz + o, fz);
        st4(dk + r * 128, ldg_if(a.pe.dK + o, fz && rin));
        st4(dbx + r * 128, ldg_if(a.pe.dbx + o, fx));
        st4(dbz + r * 128, ldg_if(a.pe.dbz + o, fz));
        p[r] = vx[r] = vz[r] = q[r] = ux[r] = uz[r] = f4(0.f);
        if (a.p0) {
            if (fx) {
                vx[r] = ld4(a.vx0 + so + o);
                ux[r] = ld4(a.ux0 + so + o);
            }
            if (fz) {
                vz[r] = ld4(a.vz0 + so + o);
                uz[r] = ld4(a.uz0 + so + o);
            }
            p[r] = ld4(p00 + e * PP + 4 * g);
            q[r] = ld4(q00 + e * PP + 4 * g);
        }
    }
    bool hsrc = false;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        hsrc |= own && sh.si[k] >= 4 * g && sh.si[k] < 4 * g + 4 && sh.sj[k] >= max(e0, 0) && sh.sj[k] < min(e0 + R, T.h);
    using Mail = ResMail<S, (CAP > 1)>;
    const Mail mb(c);
    const long long tile = (long long)T.s * c.tx * c.tz + T.t;
    unsigned long long *const boxp = a.mail + tile * mb.all, *const boxq = a.mailq + tile * mb.all;
    const long long words = (long long)c.tx * c.tz * mb.all;
    const MailSpan shotp(boxp - (long long)T.t * mb.all, words, stt), shotq(boxq - (long long)T.t * mb.all, words, stt),
        minep(boxp, mb.all, stt), mineq(boxq, mb.all, stt);
    const ResSend<S, Mail> sendp(boxp, T, c, mb, g, e0), sendq(boxq, T, c, mb, g, e0);
    const ResRecv<S, Mail> recv(T, mb, tid, nt);
    float *const prow = p00 + e0 * PP + 4 * g, *const qrow = q00 + e0 * PP + 4 * g;
    float *const vrow = &sh.vz[e0 + 2 * M][4 * lane], *const urow = &sh.uz[e0 + 2 * M][4 * lane];
    const float2 *const azr = sh.az + e0 + M, *const azhr = sh.azh + e0 + M;
    const float2 *const nc = a.st.nc;
#ifdef FWI_CHECKED
    bool sound = FWI_SPAN(sh.p, prow - (M - 1) * PP - 4, prow + (R - 1 + M) * PP + 8, stt) &&
                 FWI_SPAN(sh.q, qrow - (M - 1) * PP - 4, qrow + (R - 1 + M) * PP + 8, stt) &&
                 FWI_SPAN(sh.vz, vrow - M * PZ, vrow + (R + M - 2) * PZ + 4, stt) &&
                 FWI_SPAN(sh.uz, urow - M * PZ, urow + (R + M - 2) * PZ + 4, stt) && in_field(e0 + M, R, S::E, stt);
    for (int k = tid; k < recv.n; k += nt) {
        int w, o;
        recv.item(T, mb, k, w, o);
        sound = FWI_SPAN(sh.p, p00 + o, p00 + o + 4, stt) && FWI_SPAN(sh.q, q00 + o, q00 + o + 4, stt) && sound;
    }
    if (__syncthreads_or(!sound)) return;   // (the neighbours' waits for this tile expire)
#endif
    const bool inner = e0 >= 0 && e0 + R <= T.h;

    float wn = hsrc ? __ldg(a.src.wav + a.n0) : 0.f;
    for (int n = a.n0; n < a.n1; ++n) {
        // ---------------------------------------------------------------- velocities
        {
            float4 gp[R];
            {
                float4 w[R + HR];
#pragma unroll
                for (int k = 0; k < M - 1; ++k) w[k] = ld4(prow + (k - (M - 1)) * PP);
#pragma unroll
                for (int k = 0; k < R; ++k) w[M - 1 + k] = p[k];
#pragma unroll
                for (int k = 0; k < M; ++k) w[M - 1 + R + k] = ld4(prow + (R + k) * PP);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    gp[r] = f4(0.f);
#pragma unroll
                    for (int k = 1; k <= M; ++k) gp[r] = rtap(nc[k - 1], w[r + M - 1 + k], w[r + M - k], gp[r]);
                }
            }
            float4 w[R + HR];
#pragma unroll
            for (int k = 0; k < M - 1; ++k) w[k] = ld4(qrow + (k - (M - 1)) * PP);
#pragma unroll
            for (int k = 0; k < R; ++k) w[M - 1 + k] = q[k];
#pragma unroll
            for (int k = 0; k < M; ++k) w[M - 1 + R + k] = ld4(qrow + (R + k) * PP);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float4 gq = f4(0.f);
#pragma unroll
                for (int k = 1; k <= M; ++k) gq = rtap(nc[k - 1], w[r + M - 1 + k], w[r + M - k], gq);
                const float4 fz = rscale(azhr[r], axv);
                vz[r] = pmul(fz, pfma(bz[r], gp[r], vz[r]));
                uz[r] = pmul(fz, pfma(ld4(dbz + r * 128), gp[r], pfma(bz[r], gq, uz[r])));
                st4(vrow + r * PZ, vz[r]);
                st4(urow + r * PZ, uz[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 gpx = row_diff<M, true>(ld4(prow + r * PP - 4), p[r], ld4(prow + r * PP + 4), nc);
            const float4 gqx = row_diff<M, true>(ld4(qrow + r * PP - 4), q[r], ld4(qrow + r * PP + 4), nc);
            const float4 fx = rscale(azr[r], axhv);
            vx[r] = pmul(fx, pfma(bx[r], gpx, vx[r]));
            ux[r] = pmul(fx, pfma(ld4(dbx + r * 128), gpx, pfma(bx[r], gqx, ux[r])));
        }
        __syncthreads();
        // ------------------------------------------------------------------ pressure
        const unsigned tag = (unsigned)(n - a.n0) + 1u;
        const int slot = (n & 1) * mb.slot;
        {
            float4 dv[R];
            {
                float4 w[R + HR];
#pragma unroll
                for (int k = 0; k < M; ++k) w[k] = ld4(vrow + (k - M) * PZ);
#pragma unroll
                for (int k = 0; k < R; ++k) w[M + k] = vz[k];
#pragma unroll
                for (int k = 0; k < M - 1; ++k) w[M + R + k] = ld4(vrow + (R + k) * PZ);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float4 l, rr;
                    warp_sides<M>(vx[r], l, rr);
                    dv[r] = row_diff<M, false>(l, vx[r], rr, nc);
#pragma unroll
                    for (int k = 1; k <= M; ++k) dv[r] = rtap(nc[k - 1], w[r + M + k - 1], w[r + M - k], dv[r]);
                }
            }
            float4 w[R + HR];
#pragma unroll
            for (int k = 0; k < M; ++k) w[k] = ld4(urow + (k - M) * PZ);
#pragma unroll
            for (int k = 0; k < R; ++k) w[M + k] = uz[k];
#pragma unroll
            for (int k = 0; k < M - 1; ++k) w[M + R + k] = ld4(urow + (R + k) * PZ);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float4 l, rr;
                warp_sides<M>(ux[r], l, rr);
                float4 du = row_diff<M, false>(l, ux[r], rr, nc);
#pragma unroll
                for (int k = 1; k <= M; ++k) du = rtap(nc[k - 1], w[r + M + k - 1], w[r + M - k], du);
                const float4 fp = rscale(azr[r], axv);
                p[r] = pmul(fp, pfma(Kv[r], dv[r], p[r]));
                q[r] = pmul(fp, pfma(ld4(dk + r * 128), dv[r], pfma(Kv[r], du, q[r])));
            }
        }
        if (hsrc) {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int e = e0 + r, i = sh.si[k] - 4 * g;
                    if (sh.sj[k] == e && e >= 0 && e < T.h && i >= 0 && i < 4) {
                        add_source<true>(p[r], i, __fmul_rn(comp(Kv[r], i), wn), sh.sw[k]);
                        add_source<true>(q[r], i, __fmul_rn((dk + r * 128)[i], wn), sh.sw[k]);
                    }
                }
            if (n + 1 < a.n1) wn = __ldg(a.src.wav + n + 1);
        }
        sendp.put(T, mb, slot, e0, p, tag, shotp);
        sendq.put(T, mb, slot, e0, q, tag, shotq);
        if (own)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (inner || (e0 + r >= 0 && e0 + r < T.h)) {
                    st4(prow + r * PP, p[r]);
                    st4(qrow + r * PP, q[r]);
                }
        // ------------------------------------------------------------------ exchange
        if (e0 <= 0 && e0 + R > 0 && g == 0 && T.U && T.L) {   // the first cell of q, for the diagonal tile's samples
            float v = 0.f;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (e0 + r == 0) v = q[r].x;
            unsigned long long *const dg = boxq - (long long)(c.tx + 1) * mb.all + 2 * mb.slot + (n & 3);
            if (shotq.has(dg, 1))
                asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(dg), "l"((unsigned long long)tag << 32 | __float_as_uint(v))
                             : "memory");
        }
        bool ok = recv.get(boxp + slot, T, mb, p00, tag, tid, nt, a.wait.polls, minep);
        ok = recv.get(boxq + slot, T, mb, q00, tag, tid, nt, a.wait.polls, mineq) && ok;
        if (tid == 0 && sh.rec.diag && T.R && T.D && mineq.has(boxq + 2 * mb.slot + (n & 3), 1)) {
            unsigned long long v = 0;
            int spin = 0;
            do {
                asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(boxq + 2 * mb.slot + (n & 3)) : "memory");
            } while ((unsigned)(v >> 32) != tag && ++spin < a.wait.polls);
            ok = ok && spin < a.wait.polls;
            q00[T.h * PP + 4 * T.ng] = __uint_as_float((unsigned)v);
        }
        if (!ok) res_expired(a.wait, stt, &sh.abort);
        __syncthreads();
        if (*reinterpret_cast<volatile int *>(&sh.abort)) break;
        if (a.traces) res_sample(sh.rec, T, d, a.ridx, a.rw, a.traces, a.nr, a.nt, n, q00, PP, tid, S::E * PP - 8, stt);
        if (!own || !inner)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (!own || e0 + r < 0 || e0 + r >= T.h) {
                    p[r] = ld4(prow + r * PP);
                    q[r] = ld4(qrow + r * PP);
                }
    }
    if (a.p1)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = e0 + r, o = go + r * d.Px;
            if (FWI_IN(own && e >= 0 && e < T.h, o, 4, d.Np, stt)) {
                st4(a.p1 + so + o, p[r]);
                st4(a.vx1 + so + o, vx[r]);
                st4(a.vz1 + so + o, vz[r]);
                st4(a.q1 + so + o, q[r]);
                st4(a.ux1 + so + o, ux[r]);
                st4(a.uz1 + so + o, uz[r]);
            }
        }
}

}  // namespace fwi
