// Analysis kernels outside the step: the velocity-ellipsoid moments of the
// anisotropy analysis and the gather of a batch's records.
#pragma once
#include "m2m_kernels.cuh"

namespace m2m {

// Reciprocal of a normal double: the hardware's 20-bit approximation y and
// one third-order step, y (1 + e + e^2) with e = 1 - d y (|e| < 2^-19, so e^3
// is below half an ulp).  Three FP64 operations where a division takes
// three times as many on the pipe that bounds the kernel below.
__device__ __forceinline__ double rcp_d(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// 0, or a magnitude between 2^-400 and 2^400 (on the bits: no FP64 instruction).
__device__ __forceinline__ bool square_ok(double v) {
    const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu;
    return (hi >> 20) - 623u <= 800u || (hi | (unsigned)__double2loint(v)) == 0u;
}

// Float -> double exactly, with integer instructions for normal numbers (the
// conversion instruction runs on the FP64 pipe).
__device__ __forceinline__ double widen(float f) {
    return (__float_as_uint(f) & 0x7f800000u) - 1u < 0x7f7fffffu ? f2d_fast(f) : (double)f;
}
__device__ __forceinline__ double widen(double d) { return d; }

// Lane copies of the block's sums: lane l of every warp adds to copy
// l mod copies, so that the lanes of a warp, which mostly share a shell, do
// not queue on one address (a double shared-memory add is a compare-and-swap
// loop: 32 lanes on one sum run it 32 times).
inline int vmoments_copies(int nsh) {
    int r = 32;
    while (r > 1 && (size_t)r * 32 * nsh > 32768) r >>= 1;
    return r;
}

// Velocity-ellipsoid moments per spherical shell: lane-private double sums
// in shared memory (4 per shell and copy), one global atomic per sum and
// block.  The shell is the last edge <= r^2 (e2: the smallest values of the
// state precision >= the double edges, which is the same test), by bisection.
// v_r^2 = (x.v)^2/r^2 and v_phi^2 = (x vy - y vx)^2/R^2 come from one
// reciprocal of r^2 R^2 and no square root.  Bound by the FP64 pipe (one warp
// instruction in 16 cycles per SM): 31 of them per particle, against about
// 100 and the serialised adds before (1M particles, 8 shells: the call took
// 576 us, now 71 us).
template <class R>
__global__ void __launch_bounds__(256) k_vmoments(const R *x, const R *y, const R *z, const R *vx, const R *vy,
                                                  const R *vz, const double *w, long long n, const R *e2,
                                                  int nsh, int copies, double *out, const int *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    double *acc = (double *)smem;                           // [4 nsh][copies]
    R *ed = (R *)(acc + (size_t)4 * nsh * copies);
    for (int k = threadIdx.x; k < 4 * nsh * copies; k += blockDim.x) acc[k] = 0.0;
    for (int k = threadIdx.x; k <= nsh; k += blockDim.x) ed[k] = e2[k];
    __syncthreads();
    double *mine = acc + (threadIdx.x & (copies - 1));
    const R e_lo = ed[0], e_hi = ed[nsh];
    // the context's error word after the sums, so that the caller reads both at once
    if (blockIdx.x == 0 && threadIdx.x == 0) *(int *)(out + 4 * nsh) = *err;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const R xs = x[i], ys = y[i], zs = z[i], us = vx[i], vs = vy[i], ws = vz[i];
        const double wi = w[i];
        const R q2 = (xs * xs + ys * ys) + zs * zs;
        if (!(q2 >= e_lo && q2 < e_hi)) continue;          // outside (or NaN)
        int lo = 0, hi = nsh;                               // ed[lo] <= q2 < ed[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (ed[mid] <= q2) lo = mid; else hi = mid;
        }
        const double X = widen(xs), Y = widen(ys), Z = widen(zs), U = widen(us), V = widen(vs), W = widen(ws);
        const double R2 = fma(X, X, Y * Y), r2 = fma(Z, Z, R2);
        const double s = fma(X, U, fma(Y, V, Z * W)), t = fma(X, V, -(Y * U));
        const double v2 = fma(U, U, fma(V, V, W * W));
        // (where a square would leave the double range, the quotients before
        // the squares; on the axis v_phi = 0, at the centre v_r = 0 too)
        const bool safe = R2 > 1e-100 && r2 < 1e100 && square_ok(s) && square_ok(t);
        const double k = rcp_d(safe ? r2 * R2 : 1.0);
        double vr2 = (s * s) * (R2 * k), vp2 = (t * t) * (r2 * k);
        if (!safe) {
            const double vr = r2 > 0 ? s / sqrt(r2) : 0.0, vp = R2 > 0 ? t / sqrt(R2) : 0.0;
            vr2 = vr * vr;
            vp2 = vp * vp;
        }
        double *o = mine + 4 * lo * copies;
        atomicAdd(o, wi);
        atomicAdd(o + copies, wi * vr2);
        atomicAdd(o + 2 * copies, wi * ((v2 - vr2) - vp2));
        atomicAdd(o + 3 * copies, wi * vp2);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 4 * nsh; k += blockDim.x) {
        double v = 0.0;
        for (int c = 0; c < copies; ++c) v += acc[k * copies + ((c + k) & (copies - 1))];
        if (v != 0.0) atomicAdd(out + k, v);
    }
}

// The last record and the error word of every model of a batch into one
// array each (one thread per model).
__global__ void k_gather_records(const m2m_record *const *src, const int *const *err, int n, m2m_record *dst,
                                 int *err_out) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < n) {
        dst[m] = *src[m];
        err_out[m] = *err[m];
    }
}

// ----------------------------------------------------- particle shards
// A shard's exchange buffers after its scatter pass (one warp): the int64
// observable totals copied out (and cleared for the next scatter), the
// entropy and weight partials of the pass's blocks summed in block order,
// and, when the pass took the (E, L_z) range, the block ranges reduced to
// (min E, -max E, -max |L_z|) so that a single minimum over shards gives
// the global range.
template <class R>
__global__ void k_shard_pack(unsigned long long *y_acc, long long *totals, int nobs, const double *stat_slots,
                             int nblk, double *stats, const void *mm_slots, int mm_nblk, double *range) {
    for (int j = threadIdx.x; j < nobs; j += blockDim.x) {
        totals[j] = (long long)y_acc[j];
        y_acc[j] = 0ull;
    }
    if (threadIdx.x == 0) {
        double s = 0.0, w = 0.0;
        for (int b = 0; b < nblk; ++b) { s += stat_slots[2 * b]; w += stat_slots[2 * b + 1]; }
        stats[0] = s;
        stats[1] = w;
        if (range && mm_nblk > 0) {
            const R *mm = (const R *)mm_slots;
            double e0 = (double)mm[0], e1 = (double)mm[1], l = (double)mm[2];
            for (int b = 1; b < mm_nblk; ++b) {
                e0 = fmin(e0, (double)mm[4 * b]);
                e1 = fmax(e1, (double)mm[4 * b + 1]);
                l = fmax(l, (double)mm[4 * b + 2]);
            }
            range[0] = e0;
            range[1] = -e1;
            range[2] = -l;
        }
    }
}

// The global range back into the range slots the prior-cell pass reads
// (one slot), in the state precision (each value is one the shards' passes
// produced, so the conversion is exact).
template <class R>
__global__ void k_shard_range(const double *range, void *mm_slots) {
    R *mm = (R *)mm_slots;
    mm[0] = (R)range[0];
    mm[1] = (R)(-range[1]);
    mm[2] = (R)(-range[2]);
    mm[3] = R(0);
}

// Philox4x32-10 output words of given counters and keys, one thread per
// draw: the generator of the seeing draws, exposed for its known-answer
// check.
__global__ void k_philox_words(const unsigned *ctr, const unsigned *key, long long n, unsigned *out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 o = philox4x32_10(make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]),
                                  make_uint2(key[2 * i], key[2 * i + 1]));
    out[4 * i] = o.x;
    out[4 * i + 1] = o.y;
    out[4 * i + 2] = o.z;
    out[4 * i + 3] = o.w;
}

}  // namespace m2m
