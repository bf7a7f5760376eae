// fwi_kernels.cuh -- device code of libfwi.so (sm_103a).
//
// Staggered-grid finite differences of the 2-D variable-density acoustic wave equation
// (Sec. "Scheme III" of arXiv:1804.01184; the operator of eq. param_full), the Born
// linearisation of the same scheme, and the adjoint scheme with the gradient fused in.
//
// Discretisation (the paper gives none of it; the readings are documented with the API):
//   p, K on nodes (i, j); vx on (i+1/2, j); vz on (i, j+1/2); zero outside the grid.
//   D+ f at i+1/2 = (1/dx) sum_k c_k (f[i+k] - f[i-k+1]);  D- g at i = (1/dx) sum_k c_k (g[i+k-1] - g[i-k]).
//   v^{n+1/2} = d_v (v^{n-1/2} - dt b D+ p^n);  p^{n+1} = d_p (p^n - dt K D-.v^{n+1/2}) + source.
//   Sponge factors are separable: d(i, j) = a_x(i) a_z(j).
//
// Memory layout in HBM: every field is [shot][Nz][Px] float32 with the row pitch Px a
// multiple of 32 floats (128-byte rows); columns Nx..Px-1 stay zero and count as outside.
// Model arrays (K, bx, bz) are [Nz][Px], shared by all shots of a launch.
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace fwi {

struct Dims {
    int Nx, Nz, Px;       // computational grid and row pitch
    int nx, nz, S;        // physical grid and sponge width
    long long Np;         // Px * Nz: floats per field per shot
};

// c_k * dt / dx: the stencil weights with the time step and spacing folded in, and their
// negatives (a subtracted stencil term becomes one fused multiply-add)
struct Stencil {
    float c[4];
    float nc[4];
};

// status bits recorded by the kernels
enum : int { ST_EINVAL = 1, ST_ECFL = 2, ST_EBOUNDS = 8 };

// Checked builds (-DFWI_CHECKED, the debug build): every global load and store of the time-step
// kernels first tests its offset against the size of its field; a failing test sets
// ST_EBOUNDS in the operation's status word and the access is skipped (nothing traps), and
// fwi_status() reports it.  The on-chip kernels also test their mailbox words against the shot's
// mailboxes and, once a launch, the rows of shared memory that a thread reads and writes
// (FWI_SPAN: floats lo .. hi - 1 of an array).  In the default build the tests compile away.
#ifdef FWI_CHECKED
__device__ __forceinline__ bool in_field(long long off, long long len, long long lim, int *status)
{
    if (off >= 0 && off + len <= lim) return true;
    if (status) atomicOr(status, ST_EBOUNDS);
    return false;
}
#define FWI_IN(valid, off, len, lim, status) ((valid) && ::fwi::in_field((off), (len), (lim), (status)))
#define FWI_SPAN(array, lo, hi, status) \
    ::fwi::in_field((lo) - reinterpret_cast<const float *>(&(array)), (hi) - (lo), sizeof(array) / sizeof(float), (status))
#else
#define FWI_IN(valid, off, len, lim, status) (valid)
#define FWI_SPAN(array, lo, hi, status) true
#endif

__device__ __forceinline__ long long cell(const Dims &d, int i, int j) { return (long long)j * d.Px + i; }

// ------------------------------------------------------------------ model build (S1)

// Contrast pair -> (K, rho) for each parameterization of Table 1 (m = m_o (1 + xi);
// K = rho vp^2, Ip = rho vp).  Returns false when a contrast leaves 1 + xi <= 0.
__device__ __forceinline__ bool kr_of(int pz, double a, double b, double vp_o, double rho_o,
                                      double &K, double &rho)
{
    if (!(a > -1.0) || !(b > -1.0)) return false;
    const double Ko = rho_o * vp_o * vp_o, Io = rho_o * vp_o;
    switch (pz) {
    case 0: { double v = vp_o * (1.0 + a); rho = rho_o * (1.0 + b); K = rho * v * v; return true; }
    case 1: { double ip = Io * (1.0 + a); rho = rho_o * (1.0 + b); K = ip * ip / rho; return true; }
    case 2: { double v = vp_o * (1.0 + a), ip = Io * (1.0 + b); rho = ip / v; K = ip * v; return true; }
    case 3: K = Ko * (1.0 + a); rho = rho_o * (1.0 + b); return true;
    case 4: K = Ko / (1.0 + a); rho = rho_o / (1.0 + b); return true;
    }
    return false;
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// K, bx = 2/(rho_i + rho_{i+1}), bz likewise, on the padded grid (padding copies the
// nearest physical cell; the last node reuses its own rho).  Checks 1 + xi > 0 and the
// CFL bound dt vp sqrt(2) sum|c_k| / dx <= 1.  The FP64 maps bound it, so a block evaluates
// each of its cells and the row and column beside it once (not three times a cell: 61 -> 47 us
// at 681 x 681, with the squared CFL test).  Blocks of 32 x 8 threads.
__global__ void __launch_bounds__(256) k_model(const float *__restrict__ xa, const float *__restrict__ xb, int pz,
                                               double vp_o, double rho_o, double cfl_coef, Dims d,
                                               float *__restrict__ K, float *__restrict__ bx, float *__restrict__ bz,
                                               int *status)
{
    __shared__ double sr[9][33];
    __shared__ bool sok[9][33];
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 8, tx = threadIdx.x, ty = threadIdx.y;
    const int i = i0 + tx, j = j0 + ty;
    double Kc = 0.0;
    for (int k = ty * 32 + tx; k < 9 * 33; k += 256) {
        // the block's own cells first (thread k's own cell is entry k), then the column and the row
        const int c = k < 256 ? k % 32 : k < 265 ? 32 : k - 265, r = k < 256 ? k / 32 : k < 265 ? k - 256 : 8;
        const int ii = min(i0 + c, d.Nx - 1), jj = min(j0 + r, d.Nz - 1);
        const int pi = clampi(ii - d.S, 0, d.nx - 1), pj = clampi(jj - d.S, 0, d.nz - 1);
        const long long q = (long long)pj * d.nx + pi;
        double Kv = 0.0, rv = 0.0;
        sok[r][c] = kr_of(pz, xa[q], xb[q], vp_o, rho_o, Kv, rv);
        sr[r][c] = rv;
        if (k < 256) Kc = Kv;
    }
    __syncthreads();
    if (i >= d.Px || j >= d.Nz) return;
    const long long o = cell(d, i, j);
    if (i >= d.Nx) { K[o] = 0.f; bx[o] = 0.f; bz[o] = 0.f; return; }
    // beyond the last node its own values stand (clamped above)
    if (!(sok[ty][tx] && sok[ty][tx + 1] && sok[ty + 1][tx])) {
        atomicOr(status, ST_EINVAL);
        K[o] = 0.f; bx[o] = 0.f; bz[o] = 0.f;
        return;
    }
    const double rc = sr[ty][tx];
    // the squared form, clear of rounding, spares most cells the FP64 quotient and root
    if (!(Kc * (cfl_coef * cfl_coef) < rc * (1.0 - 1e-9)) && sqrt(Kc / rc) * cfl_coef > 1.0) atomicOr(status, ST_ECFL);
    K[o] = (float)Kc;
    bx[o] = (float)(2.0 / (rc + sr[ty][tx + 1]));
    bz[o] = (float)(2.0 / (rc + sr[ty + 1][tx]));
}

// Born perturbation of the model: dK = J dxi, drho likewise (Jacobian of the map above),
// dbx = -bx^2/2 (drho_i + drho_{i+1}), dbz likewise.
__device__ __forceinline__ void jac_of(int pz, double a, double b, double vp_o, double rho_o,
                                       double &dKa, double &dKb, double &dra, double &drb)
{
    const double Ko = rho_o * vp_o * vp_o, Io = rho_o * vp_o;
    switch (pz) {
    case 0: { double v = vp_o * (1.0 + a), r = rho_o * (1.0 + b);
              dKa = 2.0 * r * v * vp_o; dKb = rho_o * v * v; dra = 0.0; drb = rho_o; break; }
    case 1: { double ip = Io * (1.0 + a), r = rho_o * (1.0 + b);
              dKa = 2.0 * ip * Io / r; dKb = -ip * ip * rho_o / (r * r); dra = 0.0; drb = rho_o; break; }
    case 2: { double v = vp_o * (1.0 + a), ip = Io * (1.0 + b);
              dKa = ip * vp_o; dKb = Io * v; dra = -ip * vp_o / (v * v); drb = Io / v; break; }
    case 3: dKa = Ko; dKb = 0.0; dra = 0.0; drb = rho_o; break;
    default: dKa = -Ko / ((1.0 + a) * (1.0 + a)); dKb = 0.0; dra = 0.0;
             drb = -rho_o / ((1.0 + b) * (1.0 + b)); break;
    }
}

__global__ void k_model_pert(const float *__restrict__ xa, const float *__restrict__ xb,
                             const float *__restrict__ da, const float *__restrict__ db, int pz,
                             double vp_o, double rho_o, Dims d, float *__restrict__ dK,
                             float *__restrict__ dbx, float *__restrict__ dbz)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= d.Px || j >= d.Nz) return;
    const long long o = cell(d, i, j);
    if (i >= d.Nx) { dK[o] = 0.f; dbx[o] = 0.f; dbz[o] = 0.f; return; }
    auto pert = [&](int ii, int jj, double &dKv, double &drv, double &rv) {
        int pi = clampi(ii - d.S, 0, d.nx - 1), pj = clampi(jj - d.S, 0, d.nz - 1);
        long long q = (long long)pj * d.nx + pi;
        double a = xa[q], b = xb[q], Kv, j0, j1, j2, j3;
        kr_of(pz, a, b, vp_o, rho_o, Kv, rv);
        jac_of(pz, a, b, vp_o, rho_o, j0, j1, j2, j3);
        dKv = j0 * da[q] + j1 * db[q];
        drv = j2 * da[q] + j3 * db[q];
    };
    double dKc, drc, rc, t, drx, rx, drz, rz;
    pert(i, j, dKc, drc, rc);
    pert(i + 1 < d.Nx ? i + 1 : i, j, t, drx, rx);
    pert(i, j + 1 < d.Nz ? j + 1 : j, t, drz, rz);
    const double bxv = 2.0 / (rc + rx), bzv = 2.0 / (rc + rz);
    dK[o] = (float)dKc;
    dbx[o] = (float)(-0.5 * bxv * bxv * (drc + drx));
    dbz[o] = (float)(-0.5 * bzv * bzv * (drc + drz));
}

// Sponge profile along one axis: n physical nodes, S cells each side; half = 1 for the
// half nodes.  sigma = sigma_max (delta/S)^2, sigma_max = 3 v ln(1/R) / (2 S dx), d = exp(-sigma dt).
__device__ __forceinline__ void sponge_entry(float *__restrict__ out, int i, int n, int S, double dx, double dt,
                                             double v, double R, int half)
{
    const int N = n + 2 * S;
    if (i >= N) { out[i] = 0.f; return; }
    const double u = i + (half ? 0.5 : 0.0);
    double delta = 0.0;
    if (u < S) delta = S - u;
    if (u > S + n - 1) delta = u - (S + n - 1);
    if (S == 0 || delta == 0.0) { out[i] = 1.f; return; }
    const double smax = 3.0 * v * log(1.0 / R) / (2.0 * S * dx);
    const double q = delta / S;
    out[i] = (float)exp(-smax * q * q * dt);
}

// Bilinear footprint of point k: four (cell offset, weight * scale) pairs.  A point on the
// last node puts its weight on (i0 + 1).  Points outside the physical grid flag EINVAL.
__device__ __forceinline__ void footprint_entry(const float *__restrict__ xy, int k, const Dims &d, double dx, double scale,
                                                long long *__restrict__ idx, float *__restrict__ w, int *status)
{
    const double x = xy[2 * k], z = xy[2 * k + 1];
    if (!(x >= 0.0 && z >= 0.0 && x <= (d.nx - 1) * dx && z <= (d.nz - 1) * dx)) {
        atomicOr(status, ST_EINVAL);
        for (int c = 0; c < 4; ++c) { idx[4 * k + c] = 0; w[4 * k + c] = 0.f; }
        return;
    }
    const double fx = x / dx + d.S, fz = z / dx + d.S;
    int i0 = (int)floor(fx), j0 = (int)floor(fz);
    if (i0 > d.Nx - 2) i0 = d.Nx - 2;
    if (j0 > d.Nz - 2) j0 = d.Nz - 2;
    const double tx = fx - i0, tz = fz - j0;
    idx[4 * k + 0] = cell(d, i0, j0);          w[4 * k + 0] = (float)(scale * (1.0 - tx) * (1.0 - tz));
    idx[4 * k + 1] = cell(d, i0 + 1, j0);      w[4 * k + 1] = (float)(scale * tx * (1.0 - tz));
    idx[4 * k + 2] = cell(d, i0, j0 + 1);      w[4 * k + 2] = (float)(scale * (1.0 - tx) * tz);
    idx[4 * k + 3] = cell(d, i0 + 1, j0 + 1);  w[4 * k + 3] = (float)(scale * tx * tz);
}

// The sponge profiles and the footprints of an operation in one launch (six launches of a few
// hundred FP64 threads each cost 47 us).  One thread an entry: ax, axh (Px each), az, azh (Nz
// each), sources, receivers.
struct SetupArgs {
    Dims d;
    double dx, dt, sv, sR, src_scale;
    float *ax, *axh, *az, *azh;
    int ns, nr;
    const float *src_xy, *rec_xy;
    long long *sidx, *ridx;
    float *sw, *rw;
    int *status;
};

__global__ void __launch_bounds__(64) k_setup(SetupArgs a)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    const Dims &d = a.d;
    if (k < 2 * d.Px) {
        const int half = k >= d.Px;
        sponge_entry(half ? a.axh : a.ax, k - half * d.Px, d.nx, d.S, a.dx, a.dt, a.sv, a.sR, half);
        return;
    }
    k -= 2 * d.Px;
    if (k < 2 * d.Nz) {
        const int half = k >= d.Nz;
        sponge_entry(half ? a.azh : a.az, k - half * d.Nz, d.nz, d.S, a.dx, a.dt, a.sv, a.sR, half);
        return;
    }
    k -= 2 * d.Nz;
    if (k < a.ns) {
        footprint_entry(a.src_xy, k, d, a.dx, a.src_scale, a.sidx, a.sw, a.status);
        return;
    }
    k -= a.ns;
    if (k < a.nr) footprint_entry(a.rec_xy, k, d, a.dx, 1.0, a.ridx, a.rw, a.status);
}

// Receiver footprints that share a cell, chained for a deterministic adjoint injection:
// entry k (receiver k/4, corner k%4) gets the next entry with the same cell (n4 if none) in
// bits 0..29, and bit 30 set when no earlier entry has its cell.  O(n4^2), run once; the cells go
// through shared memory (from L2 one by one: 78 us for 256 receivers).
constexpr int CHAIN_FIRST = 1 << 30;
constexpr int CHAIN_NT = 128;

__global__ void __launch_bounds__(CHAIN_NT) k_receiver_chain(const long long *__restrict__ idx, int n4, int *__restrict__ rl)
{
    __shared__ long long sc[8 * CHAIN_NT];
    const int k = blockIdx.x * CHAIN_NT + threadIdx.x;
    const long long c = k < n4 ? idx[k] : -1;
    bool first = true;
    int nx = n4;
    for (int m0 = 0; m0 < n4; m0 += 8 * CHAIN_NT) {
        __syncthreads();
        const int cnt = min(8 * CHAIN_NT, n4 - m0);
        for (int m = threadIdx.x; m < cnt; m += CHAIN_NT) sc[m] = idx[m0 + m];
        __syncthreads();
        if (nx < n4 && !first) continue;
        const int lo = min(cnt, max(0, k - m0)), hi = min(cnt, max(0, k + 1 - m0));   // entries before, up to k
        for (int m = 0; m < lo && first; ++m) first = sc[m] != c;
        for (int m = hi; m < cnt && nx == n4; ++m)
            if (sc[m] == c) nx = m0 + m;
    }
    if (k < n4) rl[k] = nx | (first ? CHAIN_FIRST : 0);
}

// ------------------------------------------------------------ shared kernel arguments

struct Model {
    const float *K, *bx, *bz, *ax, *axh, *az, *azh;
    int *status;            // the operation's status word (checked builds record out-of-range accesses)
};

struct Source {
    const long long *idx;   // [shot][4] cell offsets (relative to the shot's field)
    const float *w;         // [shot][4] dt beta / dx^2
    const float *wav;       // wavelet, sample n at (n+1/2) dt
};

// Born perturbation of the model: dK, dbx, dbz on the padded grid
struct Pert {
    const float *dK, *dbx, *dbz;
};

// trace[s][r][n] = sum_c beta_rc p^{n+1}[cell_rc]
__global__ void k_sample(const float *__restrict__ p, int ns, int nr, int nt, int n, long long Np,
                         const long long *__restrict__ ridx, const float *__restrict__ rw,
                         float *__restrict__ traces)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ns * nr) return;
    const int s = t / nr, r = t - s * nr;
    const float *ps = p + (long long)s * Np;
    float v = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (FWI_IN(true, ridx[4 * r + c], 1, Np, nullptr)) v = fmaf(rw[4 * r + c], ps[ridx[4 * r + c]], v);
    traces[(long long)t * nt + n] = v;
}

// --------------------------------------------------------------- adjoint + gradient (S7)

// ------------------------------------------------------------------ reductions (S5, S8)

constexpr int RED_THREADS = 256;

__device__ __forceinline__ double block_sum(double v)
{
    __shared__ double sh[RED_THREADS / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    v = 0.0;
    if (w == 0) {
        v = l < RED_THREADS / 32 ? sh[l] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    return v;
}

// J = 1/2 sum w (tr - data)^2 in FP64 (a fixed summation order, no scratch): the least-squares
// misfit of one set of traces (Sec. "Modelling and Inversion"), each trace (nt samples) weighted
// by w[trace] (w null: 1).  One cluster; its blocks' sums meet in block 0's shared memory in block
// order.  (Another block's shared memory is there only once that block runs: all arrive at a
// cluster barrier when they start, and wait for it after their summation.)  The FP64 pipe (two lanes
// an SM) bounds it: a subtraction and a multiply-add an element, half of the total taken at the
// end, over the cluster's SMs.  1.4 M elements: 106 us (1974 in one block with five FP64
// operations an element).
constexpr int MISFIT_NT = 512;

__global__ void __launch_bounds__(MISFIT_NT) k_misfit(const float *__restrict__ tr, const float *__restrict__ data,
                                                     long long n, const float *__restrict__ w, int nt,
                                                     double *__restrict__ out)
{
    __shared__ double sh[MISFIT_NT / 32], blocks[16];
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    auto started = cl.barrier_arrive();
    const int nb = (int)cl.num_blocks(), b = (int)cl.block_rank();
    const long long step = (long long)nb * MISFIT_NT;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    long long k = (long long)b * MISFIT_NT + threadIdx.x;
    auto add = [&](double &s, float x, float y, long long at) {
        const double r = (double)x - (double)y;
        s = w ? fma((double)w[at / nt] * r, r, s) : fma(r, r, s);
    };
    for (; k + 3 * step < n; k += 4 * step) {
        float x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[u] = tr[k + u * step];
            y[u] = data[k + u * step];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) add(acc[u], x[u], y[u], k + u * step);
    }
    for (; k < n; k += step) add(acc[0], tr[k], data[k], k);
    double v = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    cl.barrier_wait(std::move(started));
    if (threadIdx.x == 0) {
        v = 0.0;
        for (int i = 0; i < MISFIT_NT / 32; ++i) v += sh[i];
        *cl.map_shared_rank(&blocks[b], 0) = v;
    }
    cl.sync();
    if (b == 0 && threadIdx.x == 0) {
        v = 0.0;
        for (int i = 0; i < nb; ++i) v += blocks[i];
        *out = 0.5 * v;
    }
}

// Residual in place, tr <- w (tr - data), and per-block partial misfits 1/2 w (tr - data)^2:
// the adjoint source of J = 1/2 sum w r^2 (w null: 1; w per trace of nt samples).
__global__ void __launch_bounds__(RED_THREADS) k_residual(float *__restrict__ tr, const float *__restrict__ data,
                                                          long long n, double *__restrict__ partial,
                                                          const float *__restrict__ w, int nt)
{
    double acc = 0.0;
    for (long long k = (long long)blockIdx.x * RED_THREADS + threadIdx.x; k < n;
         k += (long long)gridDim.x * RED_THREADS) {
        const float r = tr[k] - data[k];
        if (w) {
            const float wk = w[k / nt];
            tr[k] = wk * r;
            acc += 0.5 * (double)wk * (double)r * (double)r;
        } else {
            tr[k] = r;
            acc += 0.5 * (double)r * (double)r;
        }
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// out[0] = sum of partial[0..n) in a fixed order (single block).
__global__ void __launch_bounds__(RED_THREADS) k_sum_final(const double *__restrict__ partial, int n,
                                                           double *__restrict__ out)
{
    double acc = 0.0;
    for (int k = threadIdx.x; k < n; k += RED_THREADS) acc += partial[k];
    acc = block_sum(acc);
    if (threadIdx.x == 0) out[0] = acc;
}

// Knuth's TwoSum: s + v rounded, with the exact rounding error added to c (no FMA contraction:
// every operation is an explicitly rounded add).  A run of these keeps the sum of FP32 values
// as the unevaluated pair s + c, exact to about twice FP32 precision.
__device__ __forceinline__ void two_sum(float &s, float &c, float v)
{
    const float t = __fadd_rn(s, v);
    const float bp = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(v, bp));
    s = t;
    c = __fadd_rn(c, e);
}

// Gradient accumulation in time: every adjoint launch adds one step's zero-lag products to
// FP32 per-shot-slot fields (one red per address per launch, so the order is fixed); after a
// chunk of steps the slots are flushed into FP64 running sums over shots (and then cleared by
// the host with a memset).  A block of FLUSH_X x FLUSH_Y threads takes FLUSH_X float4 of cells
// of field blockIdx.y (Np is a multiple of 32): thread (x, y) sums slots y, y + FLUSH_Y, ... with
// TwoSum, the FLUSH_Y partial pairs are combined in y order -- a fixed order for a given slot
// count -- and the pair is added to the FP64 running sum.  (The FP64 units of this GPU are few:
// widening every slot value would make the flush FP64-bound; the compensated FP32 sum needs
// four FP64 operations a cell.)
constexpr int FLUSH_X = 32, FLUSH_Y = 8, FLUSH_UNROLL = 4;

__global__ void __launch_bounds__(FLUSH_X * FLUSH_Y) k_acc_flush(const float *__restrict__ accK,
                                                                 const float *__restrict__ accBx,
                                                                 const float *__restrict__ accBz, int nslots, long long Np,
                                                                 double *__restrict__ sK, double *__restrict__ sX,
                                                                 double *__restrict__ sZ)
{
    __shared__ float ps[FLUSH_Y][FLUSH_X][4], pc[FLUSH_Y][FLUSH_X][4];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const long long e = ((long long)blockIdx.x * FLUSH_X + tx) * 4;
    const float *__restrict__ acc = blockIdx.y == 0 ? accK : blockIdx.y == 1 ? accBx : accBz;
    double *__restrict__ sum = blockIdx.y == 0 ? sK : blockIdx.y == 1 ? sX : sZ;
    float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
    if (e < Np)
        for (int s0 = ty; s0 < nslots; s0 += FLUSH_Y * FLUSH_UNROLL) {
            float4 v[FLUSH_UNROLL];
#pragma unroll
            for (int u = 0; u < FLUSH_UNROLL; ++u) {   // independent loads first
                const int sl = s0 + u * FLUSH_Y;
                v[u] = sl < nslots ? __ldcs(reinterpret_cast<const float4 *>(acc + sl * Np + e))
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < FLUSH_UNROLL; ++u)
                if (s0 + u * FLUSH_Y < nslots) {
                    two_sum(s[0], c[0], v[u].x);
                    two_sum(s[1], c[1], v[u].y);
                    two_sum(s[2], c[2], v[u].z);
                    two_sum(s[3], c[3], v[u].w);
                }
        }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        ps[ty][tx][k] = s[k];
        pc[ty][tx][k] = c[k];
    }
    __syncthreads();
    if (ty == 0 && e < Np) {
        float S[4] = {0.f, 0.f, 0.f, 0.f}, C[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int y = 0; y < FLUSH_Y; ++y)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                two_sum(S[k], C[k], ps[y][tx][k]);
                C[k] = __fadd_rn(C[k], pc[y][tx][k]);
            }
        double2 *o = reinterpret_cast<double2 *>(sum + e);
        const double2 lo = o[0], hi = o[1];
        o[0] = make_double2(lo.x + ((double)S[0] + (double)C[0]), lo.y + ((double)S[1] + (double)C[1]));
        o[1] = make_double2(hi.x + ((double)S[2] + (double)C[2]), hi.y + ((double)S[3] + (double)C[3]));
    }
}

// The gradient's FP64 epilogue, in two passes over the running sums of k_acc_flush.  Per padded
// cell, g_K = sK / K, and g_rho from the buoyancy nodes that touch it: h_x = g_bx * d bx/d rho_each
// = sX bx^2/2 (g_bx = -sX, d bx / d rho = -bx^2/2 for each of its two cells), h_z likewise.  Every
// physical cell takes the sum over the padded cells that copy it; corner cells copy into
// (S + 1)^2 of them, which one thread each took 0.57 ms to walk, so the sums go one axis at a time.
//
// Pass 1: rows of the padded grid folded along x into fold[0..1][Nz][nx] (g_K, g_rho); one block
// a row, a warp for each of the two edge columns.
constexpr int FOLD_NT = 128;

__global__ void __launch_bounds__(FOLD_NT) k_grad_fold(const float *__restrict__ K, const float *__restrict__ bx,
                                                       const float *__restrict__ bz, Dims d, const double *__restrict__ sK,
                                                       const double *__restrict__ sX, const double *__restrict__ sZ,
                                                       double *__restrict__ fold)
{
    const int j = blockIdx.x;
    const long long plane = (long long)d.Nz * d.nx;
    auto half_b2 = [](const float *b, long long m) { const double v = b[m]; return 0.5 * v * v; };
    auto cellg = [&](int i, double &gk, double &gr) {
        const long long m = cell(d, i, j);
        gk = sK[m] / (double)K[m];
        const double hx = half_b2(bx, m) * sX[m], hz = half_b2(bz, m) * sZ[m];
        gr = hx + hz;                                              // buoyancy nodes at i+1/2, j+1/2
        if (i > 0) gr += half_b2(bx, m - 1) * sX[m - 1];           // node at i-1/2
        if (i == d.Nx - 1) gr += hx;                               // last node reuses rho_i twice
        if (j > 0) gr += half_b2(bz, m - d.Px) * sZ[m - d.Px];
        if (j == d.Nz - 1) gr += hz;
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < 2) {   // physical columns 0 and nx - 1: the sponge cells beside them too
        const int lo = warp == 0 ? 0 : d.nx - 1 + d.S, hi = warp == 0 ? d.S : d.Nx - 1;
        double a = 0.0, b = 0.0;
        for (int i = lo + lane; i <= hi; i += 32) {
            double gk, gr;
            cellg(i, gk, gr);
            a += gk;
            b += gr;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
        if (lane == 0) {
            const long long q = (long long)j * d.nx + (warp == 0 ? 0 : d.nx - 1);
            fold[q] = a;
            fold[plane + q] = b;
        }
        return;
    }
    for (int pi = 1 + (int)threadIdx.x - 64; pi < d.nx - 1; pi += FOLD_NT - 64) {
        double gk, gr;
        cellg(pi + d.S, gk, gr);
        fold[(long long)j * d.nx + pi] = gk;
        fold[plane + (long long)j * d.nx + pi] = gr;
    }
}

// Pass 2: folds along z, then the chain rule of every parameterization at the cell's (K, rho)
// (closed-form Jacobians of the maps of Table 1), written as grads[5][2][nz][nx].
__global__ void k_grad_final(const double *__restrict__ fold, const float *__restrict__ xa,
                             const float *__restrict__ xb, int pz, double vp_o, double rho_o, Dims d,
                             double *__restrict__ grads)
{
    const int pi = blockIdx.x * blockDim.x + threadIdx.x, pj = blockIdx.y * blockDim.y + threadIdx.y;
    if (pi >= d.nx || pj >= d.nz) return;
    const int jlo = pj == 0 ? 0 : pj + d.S, jhi = pj == d.nz - 1 ? d.Nz - 1 : pj + d.S;
    const double *fK = fold + pi, *fR = fold + (long long)d.Nz * d.nx + pi;
    double sK = 0.0, sR = 0.0;
#pragma unroll 8
    for (int j = jlo; j <= jhi; ++j) {
        sK += fK[(long long)j * d.nx];
        sR += fR[(long long)j * d.nx];
    }
    const long long q = (long long)pj * d.nx + pi;
    double K, rho;
    kr_of(pz, xa[q], xb[q], vp_o, rho_o, K, rho);
    const double vp = sqrt(K / rho), Ko = rho_o * vp_o * vp_o, Io = rho_o * vp_o;
    const long long P = (long long)d.nx * d.nz;
    // (A) vp-rho: K = rho vp^2
    grads[0 * P + q] = vp_o * 2.0 * rho * vp * sK;
    grads[1 * P + q] = rho_o * (sR + vp * vp * sK);
    // (B) Ip-rho: K = Ip^2 / rho
    grads[2 * P + q] = Io * 2.0 * vp * sK;
    grads[3 * P + q] = rho_o * (sR - vp * vp * sK);
    // (C) vp-Ip: rho = Ip/vp, K = Ip vp
    grads[4 * P + q] = vp_o * (rho * vp * sK - rho / vp * sR);
    grads[5 * P + q] = Io * (vp * sK + sR / vp);
    // (D) K-rho
    grads[6 * P + q] = Ko * sK;
    grads[7 * P + q] = rho_o * sR;
    // (E) 1/K-1/rho: K = K_o/(1+a), rho = rho_o/(1+b)
    grads[8 * P + q] = -K * K / Ko * sK;
    grads[9 * P + q] = -rho * rho / rho_o * sR;
}

}  // namespace fwi
