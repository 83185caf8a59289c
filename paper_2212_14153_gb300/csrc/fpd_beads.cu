// fpd_beads.cu -- the bead phase of the FPD step.
//
// One CTA, or a cluster of up to kBeadParts CTAs, per bead b (any number of
// instances in one launch):
//   Eq. 5   V_b = sum_x phi_b(x; R_b) u(x) / S_b, with u = (sum_k f_k c_k +
//           f/2) / rho and f the force density of the table that drove the
//           last collision (recomputed from that table, Eq. 4);
//   Sec 2.3 R_b <- R_b + V_b (forward Euler, dt = 1);
//   S_b = sum_x phi_b(x; R_b) at the new position (the discrete int phi_b);
// then the last CTA of an instance to finish (device-wide atomic counter, no
// waiting), or each bead's CTA of a cluster that holds the instance (kTeam),
// computes the bead forces of that instance from the new positions:
//   Eq. 11 springs, Eq. 12 bending in its general form (tangents of missing
//   segments are zero, which reproduces the edge cases of Eqs. 12b-12e),
//   plus the excluded-volume repulsion k_ev (d - r) r_hat of non-bonded beads
//   closer than d, and G = F / S for the spreading of Eq. 4.  Each bead's CTA
//   writes its place in the FP32 overlay table (positions split hi + lo) read
//   by the lattice sweep of the reduced-precision paths, with the forces the G.
//
// What bounds it: a chain of latencies.  A step of a small lattice is the
// sweep plus everything between the sweep's end and the overlay table, so
// work is moved off that chain: the bead's support cells, their profiles and
// the force density there depend only on the table of the previous step, and
// are listed in shared memory before the kernel waits for the sweep (it is
// launched while the sweep still runs).  Left on the chain are one round of
// population loads, one sum, the move, the support sum, and the forces.  us a
// step, before (list after the wait, sums in a tree, segments in FP64) and now:
// 100 x 200 with 10 beads 17.9 -> 7.4, 1024 x 256 with 20 (last CTA) 23.0 ->
// 10.6, FP64 80 x 40 with 8 153 -> 26.
//
// Sums are taken in fixed point (Fix below): exact integer additions of terms
// rounded to the point, at the scale of the largest one where it is small.  So
// they do not depend on which thread or CTA adds which cell, and a warp adds
// its lanes with redux instructions.  A bead gives the same bits in every
// launch shape (alone, in a batch, split over a cluster).
//
// Arithmetic: positions, velocities and forces of the FP64 (parity) path are
// FP64, phi evaluated exactly as a plain IEEE evaluation would; in the
// FP32/FP16-storage paths phi, u and the forces are FP32 from bead-relative
// offsets, positions and velocities FP64.  FP64 instructions are kept out of
// the reduced-precision paths' per-cell work: this GPU issues one FP64 warp
// instruction per ~16 cycles per SM.  Only beads whose support can overlap
// bead b's support are visited per cell.
#include <cuda_fp16.h>

#include <atomic>
#include <climits>
#include <type_traits>

#include "fpd_kernels.h"

namespace fpd {

namespace {

// ------------------------------------------------------- fixed-point sums
// Sum of n terms x with |x| < 2^ex as integers x 2^s, s = kTop - ex -
// ceil(log2(n + 1)): no sum can overflow, every addition is exact and order
// does not matter.  One term is rounded at 2^-(s + 1): for velocities (ex =
// kVelBits at first) over 784 box cells at 2^-41 (float) and 2^-117 (double).
// Where the largest term (mag) is so small that this is more than its own half
// ulp (below 2^-16 cells a step, 2^-63 in double), and where it does not fit
// below 2^ex, the caller repeats the sum with the ex that the largest term
// needs, so that a sum's relative accuracy does not depend on the speed.
constexpr int kVelBits = 0;
constexpr int kAgain = 4096;  // "once more with ex" is handed round as kAgain + ex, above zero
constexpr float kEarlyMove = 0.499f;
static_assert(kEarlyMove < kFastBead, "faster beads are judged by their FP64 velocity");
template <class R> struct Fix;
template <> struct Fix<float> {
    using T = long long;
    static constexpr int kTop = 50, kMantissa = 24, kLowest = -72;  // kLowest: smallest ex, |s| stays below 126
    static __device__ __forceinline__ T term(float x, int s) {
        return __float2ll_rn(x * __int_as_float((s + 127) << 23));  // |s| < 126: x scaled by 2^s
    }
    // size of |x|, ordered like |x|; the ex it needs; whether it is finite
    static __device__ __forceinline__ unsigned mag(float x) { return __float_as_uint(x) & 0x7fffffffu; }
    static __device__ __forceinline__ int need(unsigned m) { return (int)(m >> 23) - 126; }
    static __device__ __forceinline__ bool finite(unsigned m) { return m < 0x7f800000u; }
    // sum over the warp, in every lane: two pieces whose 32-lane sums fit 32 bits
    static __device__ __forceinline__ T warp_sum(T v) {
        const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x1ffffffu);
        const int b = __reduce_add_sync(0xffffffffu, (int)(v >> 25));
        return (T)b * (1 << 25) + a;
    }
};
template <> struct Fix<double> {
    using T = __int128;
    static constexpr int kTop = 126, kMantissa = 53, kLowest = -800;
    static __device__ __forceinline__ T term(double x, int s) {
        // from the bits: no FP64 instruction
        const unsigned long long u = (unsigned long long)__double_as_longlong(x);
        const int e = (int)(u >> 52) & 0x7ff;
        const unsigned long long m = (u & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
        const int sh = (e ? e : 1) - 1075 + s;
        T v = 0;
        if (sh >= 0) v = sh < 75 ? (T)m << sh : (T)0;  // a term in range has sh <= 73
        else if (sh > -64) v = (T)(m >> -sh);
        return (u >> 63) ? -v : v;
    }
    static __device__ __forceinline__ unsigned mag(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
    static __device__ __forceinline__ int need(unsigned m) { return (int)(m >> 20) - 1022; }
    static __device__ __forceinline__ bool finite(unsigned m) { return m < 0x7ff00000u; }
    static __device__ __forceinline__ T warp_sum(T v) {
        T r = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            r += (T)__reduce_add_sync(0xffffffffu, (unsigned)(v >> (26 * k)) & 0x3ffffffu) << (26 * k);
        const int c = __reduce_add_sync(0xffffffffu, (int)(v >> 104));
        return r + (T)((unsigned __int128)(T)c << 104);
    }
};
// 2^k, -1022 <= k <= 1023
__device__ __forceinline__ double pow2(int k) { return __hiloint2double((k + 1023) << 20, 0); }
// bits of n: the smallest l with n < 2^l
__device__ __forceinline__ int bit_length(int n) { return 32 - __clz(n); }

// ----------------------------------------------------------- CTA clusters
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_ctas() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// v to the place of the local shared-memory word p in the cluster's CTA `rank`
__device__ __forceinline__ void st_cluster(const void *p, unsigned rank, unsigned long long v) {
    unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
    asm volatile("mapa.shared::cluster.u32 %0, %0, %1;\n\tst.shared::cluster.u64 [%0], %2;"
                 : "+r"(a)
                 : "r"(rank), "l"(v)
                 : "memory");
}
__device__ __forceinline__ void push_cluster(const __int128 *p, unsigned rank, __int128 v) {
    st_cluster(p, rank, (unsigned long long)v);
    st_cluster(reinterpret_cast<const unsigned long long *>(p) + 1, rank, (unsigned long long)(v >> 64));
}

// Partial sums of a CTA's warps, and of the cluster's CTAs (two buffers in
// turn: a CTA may push its next partials while a slower one still reads).
template <class T, int NW> struct SumShared {
    T a[NW], b[NW];
    unsigned long long m[NW];
    T ca[2][kBeadParts], cb[2][kBeadParts];
    unsigned long long cm[2][kBeadParts];
};

// Totals of a (and b, N = 2) and the maximum of m (N = 2) over the CTA, or
// over all CTAs of its cluster; valid in every lane of warp 0.  Every thread
// calls it; use = how often this CTA has called it before (the cluster's
// first barrier phase, arrived at when the kernel starts, makes sure that
// all CTAs run).
template <class R, int NT, int N>
__device__ __forceinline__ void total(typename Fix<R>::T &a, typename Fix<R>::T &b, unsigned &m,
                                      SumShared<typename Fix<R>::T, NT / 32> &sh, int &use) {
    using F = Fix<R>;
    using T = typename F::T;
    constexpr int NW = NT / 32;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    a = F::warp_sum(a);
    if constexpr (N == 2) {
        b = F::warp_sum(b);
        m = __reduce_max_sync(0xffffffffu, m);
    }
    if (l == 0) {
        sh.a[w] = a;
        if constexpr (N == 2) {
            sh.b[w] = b;
            sh.m[w] = m;
        }
    }
    __syncthreads();
    if (w == 0) {
        a = F::warp_sum(l < NW ? sh.a[l] : (T)0);
        if constexpr (N == 2) {
            b = F::warp_sum(l < NW ? sh.b[l] : (T)0);
            m = __reduce_max_sync(0xffffffffu, l < NW ? (unsigned)sh.m[l] : 0u);
        }
    }
    if constexpr (std::is_same<R, double>::value) {
        const int parts = (int)cluster_ctas();
        if (parts > 1) {
            const int buf = use & 1;
            if (use == 0) cluster_wait();
            if (w == 0 && l < parts) {
                const unsigned me = cluster_rank();
                push_cluster(&sh.ca[buf][me], l, a);
                if constexpr (N == 2) {
                    push_cluster(&sh.cb[buf][me], l, b);
                    st_cluster(&sh.cm[buf][me], l, m);
                }
            }
            __syncwarp();
            cluster_arrive();
            cluster_wait();
            if (w == 0) {
                a = F::warp_sum(l < parts ? sh.ca[buf][l] : (T)0);
                if constexpr (N == 2) {
                    b = F::warp_sum(l < parts ? sh.cb[buf][l] : (T)0);
                    m = __reduce_max_sync(0xffffffffu, l < parts ? (unsigned)sh.cm[buf][l] : 0u);
                }
            }
        }
        ++use;
    }
}

// Release what this thread wrote and observed, add, acquire: the last
// arrival of a counter sees what the earlier ones released.
__device__ __forceinline__ unsigned arrive_acq_rel(unsigned *p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// d reduced to its nearest periodic image (period L = nx, or ny): the image
// index is found in FP32 (it is an integer) and removed exactly in FP64.
__device__ __forceinline__ double min_image(double d, int nx, float inv_nx) {
    const float k = rintf((float)d * inv_nx);
    return d - (double)k * (double)nx;
}
// the same for the y separation, applied only when y is periodic
__device__ __forceinline__ double min_image_y(const Inst &I, double d) {
    return I.periodic_y ? min_image(d, I.ny, I.f_inv_ny) : d;
}
__device__ __forceinline__ float min_image_yf(const Inst &I, float d) {
    return I.periodic_y ? d - (float)I.ny * rintf(d * I.f_inv_ny) : d;
}

// a - b of two places in [0, L] to the nearest periodic image.  The period
// comes off the larger of them, which is exact (it is between L / 2 and L), so
// that a difference across the edge is rounded at its own size and not at L's
// (an ulp of 65536 is 1/128 of a cell).
__device__ __forceinline__ float edge_diff(float a, float b, float L) {
    const float d = a - b;
    return (a - (d > 0.5f * L ? L : 0.f)) - (b - (d < -0.5f * L ? L : 0.f));
}

// A double as a pair of floats, h + l equal to it within 2^-48 of its size,
// from its bits: the conversions and subtractions are FP64 instructions, a
// chain of which took the last CTA about a microsecond.  Sizes outside
// [2^-74, 2^127) do not occur in use: 0 below, NaN above.
__device__ __forceinline__ float2 split(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(u >> 52) & 0x7ff;
    const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
    if (e < 949) return make_float2(0.f, 0.f);
    if (e >= 1150) return make_float2(__int_as_float(0x7fc00000), 0.f);
    const float h = __uint_as_float(sign | (unsigned)(e - 896) << 23 | ((unsigned)(u >> 29) & 0x7fffffu));
    const float l = (float)((unsigned)u & 0x1fffffffu) * __uint_as_float(sign | (unsigned)(e - 948) << 23);
    return make_float2(h, l);
}
// Error-free sum (Knuth): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (a + a')^2 as p + e, a' the low part of a
__device__ __forceinline__ void square2(float a, float al, float &p, float &e) {
    p = __fmul_rn(a, a);
    e = __fmaf_rn(2.0f * a, al, __fmaf_rn(a, a, -p));
}

// Length, tangent component and stretch of the segment from A to B on this
// thread's axis; the other axis' thread is the lane next to it (xor 1).
__device__ __forceinline__ void segment_axis(const Inst &I, double A, double B, double &L, double &t, double &str) {
    const double d = B - A, d2 = d * d;
    L = sqrt(d2 + __shfl_xor_sync(0xffffffffu, d2, 1));
    t = d * (1.0 / L);
    str = L - I.l0;
}
// FP32 paths: the difference of the unwrapped positions in FP64 (one
// instruction; pairs of floats of the positions themselves were 2e-9 of a cell
// off after 4096 periods of 128 columns), its square in pairs of floats
// (2^-46), as the stretch L - l0 = (|d|^2 - l0^2) / (L + l0) of a stiff spring
// is small against it and must not cancel away.
__device__ __forceinline__ void segment_axis(const Inst &I, double A, double B, float &L, float &t, float &str) {
    float dl, p, pe, s, se, q, qe;
    const float2 D = split(B - A);
    const float d = D.x + D.y;
    dl = D.y - (d - D.x);
    square2(d, dl, p, pe);
    two_sum(p, __shfl_xor_sync(0xffffffffu, p, 1), s, se);
    se += pe + __shfl_xor_sync(0xffffffffu, pe, 1);
    const float2 l0 = split(I.l0);
    square2(l0.x, l0.y, q, qe);
    L = sqrtf(s + se);
    t = d / L;
    str = ((s - q) + (se - qe)) / (L + I.f_l0);
}

// v.t of a segment from its two axes' lanes, the same in both, every rounding
// spelled out (two kernels share it).
__device__ __forceinline__ double dot_axes(double v, double t) {
    const double a = __dmul_rn(v, t);
    return __dadd_rn(a, __shfl_xor_sync(0xffffffffu, a, 1));
}
__device__ __forceinline__ float dot_axes(float v, float t) {
    const float vo = __shfl_xor_sync(0xffffffffu, v, 1), to = __shfl_xor_sync(0xffffffffu, t, 1);
    return threadIdx.x & 1 ? __fmaf_rn(vo, to, __fmul_rn(v, t)) : __fmaf_rn(v, t, __fmul_rn(vo, to));
}

// What a segment pulls its first bead with along one axis (and its second the
// other way): Eq. 11's spring, and Eq. 12's bending, k_b (t_{q+1} + t_{q-1}).
// (I - t_q t_q) / L with the tangents of missing segments zero (v their sum,
// vt = v.t).  Every rounding spelled out: two kernels share it.
__device__ __forceinline__ double segment_pull(const Inst &I, double v, double vt, double t, double str, double L) {
    const double bend = __ddiv_rn(__dmul_rn(I.k_b, __fma_rn(-vt, t, v)), L);
    return __fma_rn(__dmul_rn(I.ks_l02, str), t, -bend);
}
__device__ __forceinline__ float segment_pull(const Inst &I, float v, float vt, float t, float str, float L) {
    const float bend = __fdiv_rn(__fmul_rn(I.f_kb, __fmaf_rn(-vt, t, v)), L);
    return __fmaf_rn(__fmul_rn(I.f_ks_l02, str), t, -bend);
}

// Excluded-volume candidates of every bead of the instance into cand: beads
// that share no spring with it, nearer than l0 by an FP32 distance test with
// 1% margin.  Xf, Yf: positions relative to bead 0 of the instance.  Warp w
// of NW screens for beads w, w + NW, ..., 32 beads at a time.
template <int NW>
__device__ __forceinline__ void screen_close(const Inst &I, const float *Xf, const float *Yf, unsigned *cand) {
    const int N = I.n_beads, nb = I.nb, nw = (nb + 31) / 32;
    const int lane = threadIdx.x & 31;
    const float l0s2 = I.f_l0 * I.f_l0 * 1.0201f, fnx = (float)I.nx;
    for (int q = threadIdx.x >> 5; q < nb; q += NW) {
        const int lo = q / N * N;
        const float xq = Xf[q], yq = Yf[q];
        for (int c = 0; c < nw; ++c) {
            const int p = 32 * c + lane;
            bool near = false;
            if (p < nb) {
                float fx = xq - Xf[p];
                fx -= fnx * rintf(fx * I.f_inv_nx);
                const float fy = min_image_yf(I, yq - Yf[p]);
                const bool bonded = p == q || (p >= lo && p < lo + N && abs(p - q) < 2);
                near = fx * fx + fy * fy < l0s2 && !bonded;
            }
            const unsigned m = __ballot_sync(0xffffffffu, near);
            if (lane == 0) cand[q * nw + c] = m;
        }
    }
}

// The same for bead q of at most 32, lane p holding bead p's place.
__device__ __forceinline__ unsigned close_beads(const Inst &I, float x, float y, int q) {
    const int N = I.n_beads, p = threadIdx.x & 31, lo = q / N * N;
    float fx = __shfl_sync(0xffffffffu, x, q) - x;
    fx -= (float)I.nx * rintf(fx * I.f_inv_nx);
    const float fy = min_image_yf(I, __shfl_sync(0xffffffffu, y, q) - y);
    const bool bonded = p == q || (p >= lo && p < lo + N && abs(p - q) < 2);
    return __ballot_sync(0xffffffffu, p < I.nb && fx * fx + fy * fy < I.f_l0 * I.f_l0 * 1.0201f && !bonded);
}

// Excluded volume on bead q along axis ax (0 x, 1 y) from the beads in its
// nw candidate words, in bead order; r: interleaved x, y positions.
template <class R>
__device__ __noinline__ R close_force(const Inst &I, const double *r, const unsigned *cand, int nw, int q, int ax) {
    R f = (R)0;
    for (int c = 0; c < nw; ++c)
        for (unsigned bits = cand[c]; bits; bits &= bits - 1u) {
            const int p = 32 * c + __ffs(bits) - 1;
            const double dx = min_image(r[2 * q] - r[2 * p], I.nx, I.f_inv_nx);
            const double dy = min_image_y(I, r[2 * q + 1] - r[2 * p + 1]);
            if constexpr (std::is_same<R, double>::value) {
                const double d = sqrt(dx * dx + dy * dy);
                if (d < I.l0 && d > 0.0) f += I.k_ev * (I.l0 - d) / d * (ax ? dy : dx);
            } else {
                const float d = sqrtf((float)(dx * dx + dy * dy));
                if (d < I.f_l0 && d > 0.f) f += I.f_kev * (I.f_l0 - d) / d * (float)(ax ? dy : dx);
            }
        }
    return f;
}

// A support cell of the bead: phi of this bead, the spread force density
// there (Eq. 4 with the previous table), the cell's element offset in plane
// 0 and whether it lies in the lattice's first / last column / row (bits).
template <class R> struct alignas(16) SupportCell {
    R phi, fx, fy;
    int o, edge;
};
template <> struct alignas(16) SupportCell<float> {
    float phi, fx, fy;
    int o;
};
constexpr int kEdgeL = 1, kEdgeR = 2, kEdgeB = 4, kEdgeT = 8;
// Another bead whose support can overlap the bead's: the offset from it
// (FP32 paths) or its position (FP64), and its G.
template <class R> struct alignas(4 * sizeof(R)) Neighbour {
    R x, y, gx, gy;
};
// Box cells listed at a time (a support box of the usual beads fits at once:
// 29 x 29 cells for a = 4, xi = 1; with a CTA to an SM 45 x 45).
template <class R, int NT> struct ListCap {
    static constexpr int value = std::is_same<R, double>::value ? 1000 : NT >= 512 ? 2048 : 1280;
};

// The last CTA's view of its instance, in the shared memory the list took;
// x and y of a bead or segment side by side.
template <class R> struct ForceShared {
    double r[2 * kMaxBeads];
    R S[kMaxBeads], t[2 * kMaxBeads], pull[2 * kMaxBeads], len[kMaxBeads], str[kMaxBeads];
    float xf[kMaxBeads], yf[kMaxBeads];
    unsigned cand[kMaxBeads * (kMaxBeads / 32)];
};

// A bead's support box in the lattice: first column and row (wrapped), size,
// and the first cell's centre less the bead's position; [0] x, [1] y.
struct Support {
    int lo[2], n[2];
    float rel[2];
};
// Row and column of box cell c; rows by an FP32 reciprocal, exact below 2^19
// cells (two ulps of c / w stay below half of 1 / w), else by division.
__device__ __forceinline__ void cell_rc(const Support &b, const float inv_w, int c, int &ci, int &cj) {
    cj = inv_w != 0.0f ? (int)(((float)c + 0.5f) * inv_w) : c / b.n[0];
    ci = c - cj * b.n[0];
}
__device__ __forceinline__ float inv_width(const Support &b) {
    return b.n[0] * (int64_t)b.n[1] < (1 << 19) ? 1.0f / (float)b.n[0] : 0.0f;
}
// One axis of a support box (Support); from support_box, out of line: its
// registers are not the kernel's.
struct Axis {
    int lo, n;
    float rel;
};
__device__ __noinline__ Axis far_axis(const Inst &I, int ax, double Rx, double Ry) {
    const Box b = support_box(I, Rx, Ry);
    return Axis{ax ? b.j0 : b.i0, b.w > 0 && b.h > 0 ? (ax ? b.h : b.w) : 0,
                ax ? (float)(b.ju + 0.5 - Ry) : (float)(b.iu + 0.5 - Rx)};
}
// One axis (ax: 0 x, 1 y) of the support box of a bead at h + l on it, in
// FP32 with a cell of margin as support_box; positions of a million cells or
// more, or not finite, take support_box of the FP64 position (Rx, Ry).
__device__ __forceinline__ void support_axis(const Inst &I, int ax, float h, float l, bool far, double Rx, double Ry,
                                             int &lo, int &n, float &rel) {
    if (far) {
        const Axis f = far_axis(I, ax, Rx, Ry);
        lo = f.lo, n = f.n, rel = f.rel;
        return;
    }
    const int L = ax ? I.ny : I.nx;
    int a = (int)floorf(h - I.f_rcut - 0.5f) - 1, b = (int)ceilf(h + I.f_rcut - 0.5f) + 1;
    if (ax && !I.periodic_y) {
        a = max(a, 0);
        b = min(b, L - 1);
    } else if (b - a + 1 >= L) {
        // the whole axis: the L columns (rows) whose centres are the nearest
        // images, as the sweep takes them (phi is evaluated at these offsets)
        a = (int)ceilf((h - 0.5f - 0.5f * (float)L) + l);
        b = a + L - 1;
    }
    n = max(b - a + 1, 0);
    rel = ((float)a + 0.5f - h) - l;
    if (a < 0) a += L;
    else if (a >= L) a -= L;
    if ((unsigned)a >= (unsigned)L) a = ((a % L) + L) % L;
    lo = a;
}
__device__ __forceinline__ bool far_off(float xh, float yh) { return !(fabsf(xh) < 1.0e6f && fabsf(yh) < 1.0e6f); }

// A support box widened by one cell on every side: wrapped (x, and y when
// periodic), clipped at the walls, covering each direction at most once.
__device__ __forceinline__ Support widen(const Inst &I, Support b) {
    if (b.n[0] <= 0 || b.n[1] <= 0) return b;
    for (int ax = 0; ax < 2; ++ax) {
        const int L = ax ? I.ny : I.nx;
        if (ax && !I.periodic_y) {
            const int lo = max(b.lo[1] - 1, 0), hi = min(b.lo[1] + b.n[1], L - 1);
            b.lo[1] = lo;
            b.n[1] = hi - lo + 1;
        } else if (b.n[ax] < L) {
            b.lo[ax] = (b.lo[ax] == 0) ? L - 1 : b.lo[ax] - 1;
            b.n[ax] = min(b.n[ax] + 2, L);
        }
    }
    return b;
}

// Populations of a support cell, g_k.
template <class S, class R>
__device__ __forceinline__ void pull_support(const S *__restrict__ A, const Inst &I, const int o, const int edge,
                                             R g[9]) {
    const int x = o & 31;  // column within the strip
    if (edge == 0) {
        pull_inner<S, R>(A + o, strip_left(I, x), strip_right(I, x), I, g);
        return;
    }
    Cell C;
    C.o = o;
    const int last = col_off(I, I.nx - 1);
    C.shl = (edge & kEdgeL) ? last + 1 : strip_left(I, x);
    C.shr = (edge & kEdgeR) ? -last - 1 : strip_right(I, x);
    C.y0 = edge & kEdgeB;
    C.yn = edge & kEdgeT;
    C.bot = C.y0 && !I.periodic_y;
    C.top = C.yn && !I.periodic_y;
    pull_pops<S, R>(A, I, C, g);
}

// Resident bead CTAs per SM the reduced-precision kernels are held to (80
// registers a thread at 128 threads), so that large bead lists of a batch
// run in few waves; the FP64 parity path keeps its registers.
template <class S, int NT> struct BeadMinBlocks { static constexpr int value = 6 * kBeadThreads / NT > 1 ? 6 * kBeadThreads / NT : 2; };
template <int NT> struct BeadMinBlocks<double, NT> { static constexpr int value = 1; };

// NT threads per bead CTA: kBeadThreads for long bead lists (more CTAs
// resident), more when every bead has an SM of its own (shorter per-bead
// loops).  A cluster's CTAs (FP64) each take a share of the bead's cells.
// wait_first: wait for the sweep before listing the support (launch_beads).
// kTeam (FP32 paths, a short list of 1 to kTeamBeads beads an instance): an instance's
// CTAs form a cluster.  Each pushes its bead's new position to the others'
// shared memory while the support sums are taken and computes its own bead's
// force after one cluster barrier, instead of handing in through global memory
// to a last CTA (an atomic and a round of loads, 1.9 us, and all beads' forces
// on one SM): ten 100 x 200 instances of 10 beads 11.7 -> 10.7 us a step, one
// 9.8 -> 8.1, a 160 x 160 driven bead 10.3 -> 9.2.  The same arithmetic, so the
// same bits.
template <class S, int NT, bool kTeam>
__global__ void __launch_bounds__(NT, BeadMinBlocks<S, NT>::value)
    k_beads(const Inst *__restrict__ insts, const int4 *__restrict__ blist, const S *__restrict__ pool,
            const BeadTab tab0, const BeadTab tab1, const typename PhiArg<S>::type phi0,
            const typename PhiArg<S>::type phi1, unsigned *__restrict__ mask_write, int gparity, int advance,
            int wait_first, unsigned *__restrict__ counters, BeadExport ex, unsigned *__restrict__ status) {
    constexpr bool kF64 = std::is_same<S, double>::value;
    using R = typename std::conditional<kF64, double, float>::type;
    using F = Fix<R>;
    using T = typename F::T;
    constexpr int NW = NT / 32;
    constexpr int kCap = ListCap<R, NT>::value;
    constexpr int kPer = NT >= 512 ? 2 : 3;  // box cells a thread lists at a time
    constexpr size_t kBuf = sizeof(SupportCell<R>) * kCap > sizeof(ForceShared<R>) ? sizeof(SupportCell<R>) * kCap
                                                                                   : sizeof(ForceShared<R>);
    __shared__ Inst sI;
    __shared__ __align__(16) unsigned char s_buf[kBuf];
    __shared__ unsigned char s_edge[kF64 ? 1 : kCap];
    __shared__ Neighbour<R> s_nbr[kMaxBeads];
    __shared__ int4 s_nbox[kF64 ? kMaxBeads : 1];  // a neighbour's kept box, and where its profile starts
    __shared__ int s_noff[kF64 ? kMaxBeads : 1];
    __shared__ SumShared<T, NW> s_sum;
    __shared__ double s_R[2], s_old[2], s_S, s_unit;
    __shared__ Support s_sup;
    __shared__ unsigned s_cnt[2][NW];
    __shared__ int s_state;
    __shared__ float s_unit_f;
    __shared__ unsigned s_seen;
    SupportCell<R> *list = reinterpret_cast<SupportCell<R> *>(s_buf);

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int parts = kF64 ? (int)cluster_ctas() : 1, part = kF64 ? (int)cluster_rank() : 0;
    static_assert(!(kF64 && kTeam), "FP64 clusters share a bead");
    // team: every bead's place and whether it may be close to another
    __shared__ double s_peer[kTeam ? kTeamBeads : 1][2];
    __shared__ unsigned long long s_near[kTeam ? kTeamBeads : 1];
    if (parts > 1 || kTeam) cluster_arrive();  // waited for before the first push
    int uses = 0;
    // blist[i] = (2 slot + par_xor, global bead index, the instance's first
    // bead and bead count); NULL: instance 0, bead i
    const int it = blockIdx.x / parts;
    const int4 br = blist ? blist[it] : make_int4(0, it, 0, gridDim.x / parts);
    const int ii = br.x >> 1, b = br.y, first = br.z, nb = br.w;
    // this instance's step parity selects the table pair and the population buffer
    const int parity = gparity ^ (br.x & 1);
    const BeadTab &told = parity ? tab0 : tab1;
    const BeadTab &tnew = parity ? tab1 : tab0;
    const typename PhiArg<S>::type &pold = parity ? phi0 : phi1, &pnew = parity ? phi1 : phi0;
    if (advance && wait_first) {
        pdl_wait();
        pdl_trigger();
    }
    {
        // asynchronous copy of the instance record, 8 bytes a thread (a plain
        // copy's stores would hold back the loads below until it arrived)
        static_assert(sizeof(Inst) % 8 == 0 && alignof(Inst) == 8, "Inst is copied 8 bytes at a time");
        for (int wd = tid; wd < (int)(sizeof(Inst) / 8); wd += NT)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                             static_cast<unsigned>(__cvta_generic_to_shared((uint64_t *)&sI + wd))),
                         "l"((const uint64_t *)(insts + ii) + wd)
                         : "memory");
    }
    auto record_here = []() {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    };
    // Up to pdl_wait() only the records and the old table are read: the
    // preceding launch, a sweep, may still be running, but it was released
    // after the bead phase that wrote this table had completed (its lead CTA
    // waits for it).  Table reads go to L2 (an SM's L1 may hold lines of an
    // earlier step).
    int any_close = 0;  // some bead may come within the excluded volume's reach of this one
    double S_old = 1.0;  // the bead's old support sum
    float xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f;
    if (advance) {
        xh = __ldcg(told.xh + b);
        xl = __ldcg(told.xl + b);
        yh = __ldcg(told.yh + b);
        yl = __ldcg(told.yl + b);
        // and its old position, in shared memory (FP64 registers are dear)
        if (tid < 2) s_old[tid] = __ldcg((tid ? told.Ry : told.Rx) + b);
        if (tid == NT - 1) S_old = __ldcg(told.S + b);
    }
    // the lattice cell of row cj, column ci of a support box
    auto cell_of = [](const Inst &I, const Support &bx, int ci, int cj, int &i, int &j) {
        j = bx.lo[1] + cj;
        j = (j >= I.ny) ? j - I.ny : j;
        i = bx.lo[0] + ci;
        i = (i >= I.nx) ? i - I.nx : i;
    };
    const Inst &I = sI;
    if (advance) {
        // beads whose support can overlap b's (FP32 screen, 1-cell margin),
        // in bead order; every warp screens all of them, 32 at a time, so
        // that no barrier is needed, and warp 0 lists them
        int nn = 0, self = 0;  // neighbours, the bead's own place among them
        int fiber = 0;         // first bead of its fiber
        for (int q0 = 0; q0 < nb; q0 += 32) {
            const int q = q0 + lane, gq = first + q;
            float qx = 0.f, qy = 0.f;
            Neighbour<R> nbr{};
            int4 qbox = make_int4(0, 0, 0, 0);
            if (q < nb) {
                qx = __ldcg(told.xh + gq);
                const float lx = xl - __ldcg(told.xl + gq);
                qy = __ldcg(told.yh + gq);
                const float ly = yl - __ldcg(told.yl + gq);
                if constexpr (kF64) {
                    if (pold.box) qbox = __ldcg(pold.box + gq);
                    nbr.x = __ldcg(told.Rx + gq);
                    nbr.y = __ldcg(told.Ry + gq);
                    nbr.gx = __ldcg(told.Gx + gq);
                    nbr.gy = __ldcg(told.Gy + gq);
                } else {
                    nbr.x = lx;
                    nbr.y = ly;
                    nbr.gx = __ldcg(told.gxf + gq);
                    nbr.gy = __ldcg(told.gyf + gq);
                }
            }
            if (q0 == 0) record_here();
            // nearest image of the bead from bead q, by the high parts
            const float dx = edge_diff(xh, qx, (float)I.nx);
            const float dy = I.periodic_y ? edge_diff(yh, qy, (float)I.ny) : yh - qy;
            const float d2 = dx * dx + dy * dy, reach = 2.0f * I.f_rcut + 1.0f;
            const bool hit = q < nb && (d2 < reach * reach || gq == b);  // itself even if not finite
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            // two beads that move less than half a cell per component come
            // at most 1.42 cells nearer in this phase
            const float lim = I.f_l0 + 1.5f;
            if (q0 == 0) fiber = (b - first) / I.n_beads * I.n_beads;
            const bool bonded = abs(gq - b) < 2 && q >= fiber && q < fiber + I.n_beads;
            any_close |= __any_sync(0xffffffffu, q < nb && !bonded && d2 < lim * lim);
            const int lb = b - first - q0;
            if ((unsigned)lb < 32u) self = nn + __popc(m & ((1u << lb) - 1u));
            if (hit && w == 0) {
                const int pos = nn + __popc(m & ((1u << lane) - 1u));
                if constexpr (!kF64) {
                    nbr.x += dx;
                    nbr.y += dy;
                }
                s_nbr[pos] = nbr;
                if constexpr (kF64) {
                    s_nbox[pos] = qbox;
                    s_noff[pos] = I.phi_off + q * I.phi_cap;
                }
            }
            nn += __popc(m);
        }
        if constexpr (kF64) __syncthreads();  // the neighbours are in place (FP32: make_list's first barrier)
        // populations are pulled from the current buffer
        const S *A = pop_buffer(pool, I, parity);
        const bool kept = kF64 && I.phi_cap != 0;
        Support bx;
        if (kept) {
            const int4 kb = s_nbox[self];
            bx.lo[0] = kb.x, bx.lo[1] = kb.y;
            bx.n[0] = kb.z, bx.n[1] = kb.w;
        } else {
            const bool far = far_off(xh, yh);
            support_axis(I, 0, xh, xl, far, s_old[0], s_old[1], bx.lo[0], bx.n[0], bx.rel[0]);
            support_axis(I, 1, yh, yl, far, s_old[0], s_old[1], bx.lo[1], bx.n[1], bx.rel[1]);
        }
        const float inv_w = inv_width(bx);
        // List the support cells (phi_b != 0) among box cells [c0, c1),
        // c1 - c0 <= kCap, with the force density of the previous table.
        auto make_list = [&](int c0, int c1) -> int {
            int n = 0;
#pragma unroll 1
            for (int r0 = c0, buf = 0; r0 < c1; r0 += kPer * NT, buf ^= 1) {
                // kPer cells a thread: independent evaluations in flight
                R ph[kPer];
                unsigned m[kPer], cnt = 0u;
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const int c = r0 + k * NT + tid;
                    ph[k] = (R)0;
                    if (c < c1) {
                        int ci, cj;
                        cell_rc(bx, inv_w, c, ci, cj);
                        if constexpr (kF64) {
                            if (kept) {
                                ph[k] = __ldcg(pold.phi + s_noff[self] + c);
                            } else {
                                int i, j;
                                cell_of(I, bx, ci, cj, i, j);
                                ph[k] = phi_f64(I, i + 0.5, j + 0.5, s_old[0], s_old[1]);
                            }
                        } else {
                            ph[k] = phi_f32(bx.rel[0] + (float)ci, bx.rel[1] + (float)cj, I.f_a, I.f_inv_xi, I.f_rcut2);
                        }
                    }
                    m[k] = __ballot_sync(0xffffffffu, ph[k] != (R)0);
                    cnt += __popc(m[k]);
                }
                // places: after the cells of the warps before this one
                if (lane == 0) s_cnt[buf][w] = cnt;
                __syncthreads();
                const unsigned of = lane < NW ? s_cnt[buf][lane] : 0u;
                int at = n + (int)__reduce_add_sync(0xffffffffu, lane < w ? of : 0u);
                n += (int)__reduce_add_sync(0xffffffffu, of);
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    if (ph[k] != (R)0) {
                        SupportCell<R> &sc = list[at + __popc(m[k] & ((1u << lane) - 1u))];
                        sc.phi = ph[k];
                        sc.o = r0 + k * NT + tid;
                    }
                    at += __popc(m[k]);
                }
            }
            __syncthreads();
            // entries tid, tid + NT, ... are read back by this thread only
#pragma unroll 1
            for (int e = tid; e < n; e += NT) {
                int ci, cj, i, j;
                cell_rc(bx, inv_w, list[e].o, ci, cj);
                cell_of(I, bx, ci, cj, i, j);
                R fx, fy;
                if constexpr (kF64) {
                    fx = I.gx, fy = I.gy;
                    if (kept) {
#pragma unroll 4
                        for (int q = 0; q < nn; ++q) {
                            const int at = box_place(I, s_nbox[q], i, j);
                            const double ph = at >= 0 ? __ldcg(pold.phi + s_noff[q] + at) : 0.0;
                            fx += ph * s_nbr[q].gx;
                            fy += ph * s_nbr[q].gy;
                        }
                    } else {
#pragma unroll 1
                        for (int q = 0; q < nn; ++q) {
                            const double ph = phi_f64(I, i + 0.5, j + 0.5, s_nbr[q].x, s_nbr[q].y);
                            fx += ph * s_nbr[q].gx;
                            fy += ph * s_nbr[q].gy;
                        }
                    }
                } else {
                    const float own = list[e].phi;
                    const float hnx = 0.5f * (float)I.nx, fnx = (float)I.nx;
                    const float hny = 0.5f * (float)I.ny, fny = (float)I.ny;
                    const float dx = bx.rel[0] + (float)ci, dy = bx.rel[1] + (float)cj;
                    fx = I.f_gx, fy = I.f_gy;
#pragma unroll 2
                    for (int q = 0; q < nn; ++q) {
                        const Neighbour<R> nbr = s_nbr[q];
                        float ddx = dx + nbr.x;
                        ddx = (ddx > hnx) ? ddx - fnx : ((ddx < -hnx) ? ddx + fnx : ddx);
                        float ddy = dy + nbr.y;
                        if (I.periodic_y) ddy = (ddy > hny) ? ddy - fny : ((ddy < -hny) ? ddy + fny : ddy);
                        const float ph = q == self ? own : phi_f32(ddx, ddy, I.f_a, I.f_inv_xi, I.f_rcut2);
                        fx += ph * nbr.gx;
                        fy += ph * nbr.gy;
                    }
                }
                list[e].fx = fx;
                list[e].fy = fy;
                list[e].o = j * kRowStride + col_off(I, i);
                const int edge = (i == 0 ? kEdgeL : 0) | (i == I.nx - 1 ? kEdgeR : 0) | (j == 0 ? kEdgeB : 0) |
                                 (j == I.ny - 1 ? kEdgeT : 0);
                if constexpr (kF64) list[e].edge = edge;
                else s_edge[e] = (unsigned char)edge;
            }
            return n;
        };
        const int ncell = bx.n[0] * bx.n[1], share = (ncell + parts - 1) / parts;
        const int c_lo = min(part * share, ncell), c_hi = min(c_lo + share, ncell);
        if (tid == NT - 1) {
            s_unit = 1.0 / S_old * pow2(-(F::kTop - kVelBits - bit_length(ncell)));
            s_unit_f = (float)s_unit;
        }
        int n = make_list(c_lo, min(c_lo + kCap, c_hi));
        // wait for the preceding sweep (the populations read below), then let
        // the next sweep launch at once: its tiles that no bead marked start
        // while the rest of this phase runs
        if (!wait_first) {
            pdl_wait();
            pdl_trigger();
        }
        // a largest term that needs less is rounded by the sum (once more, then)
        int least = kVelBits - (F::kTop - F::kMantissa - bit_length(ncell));
#pragma unroll 1
        for (int bound = kVelBits;;) {
            const int s = F::kTop - bound - bit_length(ncell);
            T ax = 0, ay = 0;
            unsigned mx = 0u;
#pragma unroll 1
            for (int c0 = c_lo;;) {
#pragma unroll 1
                for (int e = tid; e < n; e += NT) {
                    const SupportCell<R> sc = list[e];
                    int edge;
                    if constexpr (kF64) edge = sc.edge;
                    else edge = s_edge[e];
                    R g[9];
                    pull_support<S, R>(A, I, sc.o, edge, g);
                    R ux, uy;
                    if constexpr (kF64) {
                        double dr = 0.0;
#pragma unroll
                        for (int k = 0; k < 9; ++k) dr += g[k];
                        const double rho = 1.0 + dr;
                        const double jx = g[1] - g[3] + g[5] - g[6] - g[7] + g[8];
                        const double jy = g[2] - g[4] + g[5] + g[6] - g[7] - g[8];
                        ux = (jx + 0.5 * sc.fx) / rho;
                        uy = (jy + 0.5 * sc.fy) / rho;
                    } else {
                        const float rho =
                            1.0f + (((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8]);
                        const float jx = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
                        const float jy = (g[2] - g[4]) + (g[5] + g[6]) - (g[7] + g[8]);
                        const float irho = __frcp_rn(rho);
                        ux = (jx + 0.5f * sc.fx) * irho;
                        uy = (jy + 0.5f * sc.fy) * irho;
                    }
                    const R tx = sc.phi * ux, ty = sc.phi * uy;
                    ax += F::term(tx, s);
                    ay += F::term(ty, s);
                    mx = max(mx, max(F::mag(tx), F::mag(ty)));
                }
                c0 += kCap;
                if (c0 >= c_hi) break;
                __syncthreads();  // the list is no longer read
                n = make_list(c0, min(c0 + kCap, c_hi));
            }
            total<R, NT, 2>(ax, ay, mx, s_sum, uses);
            // FP32 paths: the new support box from the old place and V in FP32,
            // a few instructions, so that the support sum need not wait for
            // the FP64 chain of the move (FP64 instructions cost a warp 64
            // cycles or more each): V clearly below kFastBead, whose rounding
            // (2^-25) is far below the box offsets' own
            if (w == 0) {
                const int need = F::need(mx);
                // a term of magnitude 2^kVelBits or more (a diverging run), or
                // all of them so small that they were rounded: once more
                int state = -1;
                if ((need > bound || need < least) && mx != 0u && F::finite(mx)) state = kAgain + max(need, F::kLowest);
                if constexpr (!kF64) {
                    const float vx = (float)ax * s_unit_f, vy = (float)ay * s_unit_f;
                    if (state < 0 && bound <= kVelBits && F::finite(mx) && fabsf(vx) < kEarlyMove && fabsf(vy) < kEarlyMove &&
                        !far_off(xh, yh)) {
                        state = 0;
                        if (lane < 2)
                            support_axis(I, lane, lane ? yh : xh, lane ? yl + vy : xl + vx, false, 0.0, 0.0,
                                         s_sup.lo[lane], s_sup.n[lane], s_sup.rel[lane]);
                    }
                }
                if (lane == 0) s_state = state;
            }
            __syncthreads();
            const int state = s_state;
            if (state > 0) {
                bound = state - kAgain;
                least = INT_MIN;
                if constexpr (!kF64)
                    if (tid == 0 && bound < kVelBits) s_unit_f *= __int_as_float((bound - kVelBits + 127) << 23);
                if (c_hi - c_lo > kCap) n = make_list(c_lo, min(c_lo + kCap, c_hi));  // else it is still in place
                continue;
            }
            if constexpr (kTeam) cluster_wait();  // the cluster's CTAs all run
            if (w == 0) {
                // the move; lane 0: x, the others: y
                double unit = s_unit;
                if (bound != kVelBits) unit *= pow2(bound - kVelBits);
                double v = (double)(lane == 0 ? ax : ay) * unit;
                if (!F::finite(mx)) v = __longlong_as_double(0x7ff8000000000000ll);
                const double r = s_old[lane == 0 ? 0 : 1] + v;
                if (part == 0 && lane < 2) {
                    (lane ? tnew.Ry : tnew.Rx)[b] = r;
                    (lane ? tnew.Vy : tnew.Vx)[b] = v;
                }
                if (lane < 2) s_R[lane] = r;
                if (state < 0) {
                    const float h = (float)r, l = (float)(r - (double)h);
                    const double rx = __shfl_sync(0xffffffffu, r, 0), ry = __shfl_sync(0xffffffffu, r, 1);
                    const bool far = far_off(__shfl_sync(0xffffffffu, h, 0), __shfl_sync(0xffffffffu, h, 1));
                    if (lane < 2) support_axis(I, lane, h, l, far, rx, ry, s_sup.lo[lane], s_sup.n[lane], s_sup.rel[lane]);
                    // fast-bead guard (below): this bead's bits, |v| >=
                    // kFastBead or not finite by the high word
                    const unsigned hv = (unsigned)__double2hiint(v) & 0x7fffffffu;
                    const bool fast = hv >= (unsigned)__double2hiint(kFastBead);
                    any_close |= __any_sync(0xffffffffu, fast);
                    if (part == 0 && lane < 2 && status && fast)
                        atomicOr(status + ii, kFlagFastBead | (hv >= 0x7ff00000u ? kFlagNonFinite : 0u));
                }
                if constexpr (kTeam) {
                    const double ra = __shfl_sync(0xffffffffu, r, lane & 1);
                    if (lane < 2 * nb)
                        st_cluster(&s_peer[b - first][lane & 1], lane >> 1, (unsigned long long)__double_as_longlong(ra));
                    if (lane < nb) st_cluster(&s_near[b - first], lane, any_close ? 1ull : 0ull);
                }
            }
            if (state < 0) __syncthreads();
            break;
        }
    } else {
        pdl_wait();
        pdl_trigger();
        record_here();
        any_close = 1;
        if (tid < 2) {
            const double rx = tnew.Rx[b], ry = tnew.Ry[b], r = tid ? ry : rx;
            const float h = (float)r;
            support_axis(I, tid, h, (float)(r - (double)h), far_off((float)rx, (float)ry), rx, ry, s_sup.lo[tid],
                         s_sup.n[tid], s_sup.rel[tid]);
            s_R[tid] = r;
        }
        __syncthreads();
    }

    // S_b = sum_x phi_b at the new position
    T acc = 0, none = 0;
    unsigned mx = 0u;
    const Support bx = s_sup;
    const float inv_w = inv_width(bx);
    const int ncell = bx.n[0] * bx.n[1], share = (ncell + parts - 1) / parts;
    const int c_lo = min(part * share, ncell), c_hi = min(c_lo + share, ncell);
    const int s_shift = F::kTop - 1 - bit_length(ncell);  // phi < 2
#pragma unroll 1
    for (int c = c_lo + (tid + NT - 32) % NT; c < c_hi; c += NT) {  // warp 0, busy with the move, comes last
        R ph;
        int ci, cj;
        cell_rc(bx, inv_w, c, ci, cj);
        if constexpr (kF64) {
            int i, j;
            cell_of(I, bx, ci, cj, i, j);
            ph = phi_f64(I, i + 0.5, j + 0.5, s_R[0], s_R[1]);
        } else {
            ph = phi_f32(bx.rel[0] + (float)ci, bx.rel[1] + (float)cj, I.f_a, I.f_inv_xi, I.f_rcut2);
        }
        acc += F::term(ph, s_shift);
        if constexpr (kF64) {
            // kept for the sweep and the next bead phase; a box has at most phi_cap cells
            if (c < I.phi_cap) pnew.phi[I.phi_off + (b - first) * I.phi_cap + c] = ph;
        }
    }
    if constexpr (kF64) {
        if (I.phi_cap && part == 0 && tid == 0) pnew.box[b] = make_int4(bx.lo[0], bx.lo[1], bx.n[0], bx.n[1]);
    }
    if constexpr (kTeam) {
        __syncwarp();
        cluster_arrive();  // this CTA's pushes (warp 0) are done
    }
    total<R, NT, 1>(acc, none, mx, s_sum, uses);
    if (part != 0) return;

    // The last CTA of this instance computes the forces of all its beads:
    // warp 0 hands in the bead (R, V and S) while the others mark tiles.  An
    // arrival counts 1, and 2^16 if the excluded volume may act on the bead.
    if (w == 0) {
        if (lane == 0) s_S = tnew.S[b] = (double)acc * pow2(-s_shift);
        if constexpr (!kTeam) {
            __syncwarp();  // lane 1's R and V before lane 0's release
            if (lane == 0) {
                s_seen = 0u;
                if (nb > 1)
                    s_seen = arrive_acq_rel(&counters[ii], any_close ? 0x10001u : 1u) | (any_close ? 0x10000u : 0u);
            }
        }
    } else {
        // FP32 overlay table: x (and y when periodic) wrapped into the
        // lattice, split into hi + lo
        if (w == 1 && lane < 2) {
            double v = s_R[lane];
            if (lane == 0 || I.periodic_y) {
                const int L = lane ? I.ny : I.nx;
                v -= (double)floorf((float)v * (lane ? I.f_inv_ny : I.f_inv_nx)) * (double)L;
                v = (v < 0.0) ? v + L : ((v >= L) ? v - L : v);
            }
            const float hi = (float)v;
            (lane ? tnew.yh : tnew.xh)[b] = hi;
            (lane ? tnew.yl : tnew.xl)[b] = (float)(v - (double)hi);
        }
        // mark bead b in the mask of every lattice tile its support box, widened
        // by one cell, reaches (the part before a periodic edge, then the part
        // after it; a tile reached twice is marked twice); the widening covers
        // the bead's move in the next step, so the next sweep may update
        // unmarked tiles before its bead phase ends
        const Support wb = widen(I, bx);
        const int lb = b - first;
        const unsigned bit = 1u << (lb & 31);
        const int c0 = wb.lo[0] / kTileX, c1 = (min(wb.lo[0] + wb.n[0], I.nx) - 1) / kTileX;
        const int r0 = wb.lo[1] / kTileY, r1 = (min(wb.lo[1] + wb.n[1], I.ny) - 1) / kTileY;
        const int over_x = wb.lo[0] + wb.n[0] - I.nx, over_y = wb.lo[1] + wb.n[1] - I.ny;
        const int nc = c1 - c0 + 1, cols = nc + (over_x > 0 ? (over_x - 1) / kTileX + 1 : 0);
        const int nr = r1 - r0 + 1, rows = nr + (over_y > 0 ? (over_y - 1) / kTileY + 1 : 0);
        const int marks = wb.n[0] > 0 && wb.n[1] > 0 ? rows * cols : 0;
#pragma unroll 1
        for (int t = tid - 32; t < marks; t += NT - 32) {
            const int tr = t / cols, tc = t - tr * cols;
            const int row = tr < nr ? r0 + tr : tr - nr, col = tc < nc ? c0 + tc : tc - nc;
            const int tile = I.tile_base + row * I.ntx + col;
            atomicOr(mask_write + tile * I.mask_words + (lb >> 5), bit);
        }
    }
    if constexpr (kTeam) {
        const int q = b - first, N = I.n_beads, i0 = q - N * (int)(((float)q + 0.5f) * (1.0f / (float)N));
        cluster_wait();  // every bead's place is here, and its status bits are set
        // fast-bead guard, as below
        if (w != 0) {
            if (q == 0 && status && (__ldcg(status + ii) & kFlagFastBead))
                for (int t = tid - 32; t < I.ntx * I.nty; t += NT - 32)
                    atomicOr(mask_write + (I.tile_base + t) * I.mask_words, 1u);
            return;
        }
        const bool crowd = I.k_ev != 0.0 && __any_sync(0xffffffffu, lane < nb && s_near[lane] != 0ull);
        // lanes 2 m + ax, m < 4: axis ax of segment q - 2 + m of the fiber
        const int ax = lane & 1, m = (lane >> 1) & 3, j = q - 2 + m;
        const bool seg = i0 - 2 + m >= 0 && i0 - 2 + m < N - 1;
        float f = 0.f;  // in lanes 4 and 5 (m = 2)
        if (N > 1) {
            float L, t, str;
            segment_axis(I, s_peer[seg ? j : 0][ax], s_peer[seg ? j + 1 : 0][ax], L, t, str);
            if (!seg) t = 0.f;
            const float tn = __shfl_down_sync(0xffffffffu, t, 2), tp = __shfl_up_sync(0xffffffffu, t, 2);
            const float v = tn + tp, vt = dot_axes(v, t);
            const float pull = seg ? segment_pull(I, v, vt, t, str, L) : 0.f;
            const float before = __shfl_up_sync(0xffffffffu, pull, 2);
            if (i0 > 0) f -= before;
            if (i0 < N - 1) f += pull;
        }
        if (crowd) {
            const int p = lane < nb ? lane : 0;
            const float x = (float)(s_peer[p][0] - s_peer[0][0]), y = (float)(s_peer[p][1] - s_peer[0][1]);
            const unsigned cand = close_beads(I, x, y, q);
            f += close_force<float>(I, &s_peer[0][0], &cand, 1, q, ax);
        }
        f += ax ? I.f_ext_fy : I.f_ext_fx;
        if ((lane >> 1) == 2) {
            const float g = f * (1.0f / (float)s_S);
            (ax ? tnew.gyf : tnew.gxf)[b] = g;
            (ax ? tnew.Gy : tnew.Gx)[b] = g;
            (ax ? tnew.Fy : tnew.Fx)[b] = f;
        }
        return;
    }
    __syncthreads();
    const unsigned seen = s_seen;  // arrivals before this one, and this one's flag
    if ((seen & 0xffffu) != (unsigned)(nb - 1)) return;
    const bool crowd = I.k_ev != 0.0 && (seen >> 16) != 0u;
    ForceShared<R> &fs = *reinterpret_cast<ForceShared<R> *>(s_buf);
    // this phase's export number (the previous phase wrote the counter)
    const unsigned long long ex_k = ex.ring ? *(volatile unsigned long long *)ex.count : 0ull;
    // the instance's status bits, this phase's among them
    const unsigned st_now = (status && advance) ? __ldcg(status + ii) : 0u;
    // The instance's new positions and support sums (written by every CTA;
    // the L2-coherent loads see them), then every segment, then every bead;
    // a thread works on one axis (ax) of item q (FP64 instructions cost a
    // warp 64 cycles each whatever its lanes do, so x and y share them)
    const int items = 2 * nb, N = I.n_beads;
    const float inv_n = 1.0f / (float)N;
    for (int k = tid; k < items; k += NT) {
        fs.r[k] = nb == 1 ? s_R[k] : __ldcg(((k & 1) ? tnew.Ry : tnew.Rx) + first + (k >> 1));
        if (!(k & 1)) fs.S[k >> 1] = (R)(nb == 1 ? s_S : __ldcg(tnew.S + first + (k >> 1)));
    }
    __syncthreads();
    // fast-bead guard: the early update of unmarked tiles assumes a bead
    // moves less than a cell per step.  When a velocity has reached kFastBead
    // per component (or is not finite) the instance is flagged; while the
    // flag is set, mark every tile of the instance (bead 0's bit) in this
    // phase's masks, so that the next sweeps wait on all of them
    if (st_now & kFlagFastBead)
        for (int t = tid; t < I.ntx * I.nty; t += NT) atomicOr(mask_write + (I.tile_base + t) * I.mask_words, 1u);
    // place of bead q < 256 within its fiber
    auto in_fiber = [&](int q) { return q - N * (int)(((float)q + 0.5f) * inv_n); };
    // Segment q (bead q to q + 1 of the fiber): length, tangent, stretch
    for (int k0 = 0; k0 < items; k0 += NT) {
        const int k = k0 + tid, q = k >> 1;
        const bool seg = k < items && in_fiber(q) < N - 1;
        R L, t, str;
        segment_axis(I, fs.r[seg ? k : 0], fs.r[seg ? k + 2 : 1], L, t, str);
        if (seg) {
            fs.t[k] = t;
            if (!(k & 1)) {
                fs.len[q] = L;
                fs.str[q] = str;
            }
        }
    }
    if (crowd) {
        for (int q = tid; q < nb; q += NT) {
            fs.xf[q] = (float)(fs.r[2 * q] - fs.r[0]);
            fs.yf[q] = (float)(fs.r[2 * q + 1] - fs.r[1]);
        }
        __syncthreads();
        screen_close<NW>(I, fs.xf, fs.yf, fs.cand);
    }
    __syncthreads();
    // What segment q pulls bead q with
    for (int k0 = 0; k0 < items; k0 += NT) {
        const int k = k0 + tid, q = k >> 1, i0 = in_fiber(q);
        const bool seg = k < items && i0 < N - 1;
        R v = (R)0, t = (R)0;
        if (seg) {
            t = fs.t[k];
            if (i0 < N - 2) v = fs.t[k + 2];
            if (i0 > 0) v += fs.t[k - 2];
        }
        const R vt = dot_axes(v, t);
        if (seg) fs.pull[k] = segment_pull(I, v, vt, t, fs.str[q], fs.len[q]);
    }
    __syncthreads();
    for (int k = tid; k < items; k += NT) {
        const int q = k >> 1, ax = k & 1, gq = first + q, i0 = in_fiber(q);
        R f = (R)0;
        if (i0 > 0) f -= fs.pull[k - 2];
        if (i0 < N - 1) f += fs.pull[k];
        if (crowd) f += close_force<R>(I, fs.r, fs.cand + q * ((nb + 31) / 32), (nb + 31) / 32, q, ax);
        // constant external force F_0 (driven particle, Sec. 3.2)
        if constexpr (kF64) f += ax ? I.ext_fy : I.ext_fx;
        else f += ax ? I.f_ext_fy : I.f_ext_fx;
        R g;
        g = f * ((R)1 / fs.S[q]);
        (ax ? tnew.gyf : tnew.gxf)[gq] = (float)g;
        (ax ? tnew.Gy : tnew.Gx)[gq] = g;
        (ax ? tnew.Fy : tnew.Fx)[gq] = f;
        if (ex.ring) {
            // export: R, V, F, S of bead q into the ring slot of this phase
            double *d = ex.ring + (size_t)(ex_k % (unsigned long long)ex.slots) * ex.stride + kExportHeader;
            d[ax * nb + q] = __ldcg((ax ? tnew.Ry : tnew.Rx) + gq);
            d[(2 + ax) * nb + q] = __ldcg((ax ? tnew.Vy : tnew.Vx) + gq);
            d[(4 + ax) * nb + q] = f;
            if (!ax) d[6 * nb + q] = __ldcg(tnew.S + gq);
        }
    }
    if (ex.ring) {
        // the table is in host memory before its slot header says so
        __threadfence_system();
        __syncthreads();
        if (tid == 0) {
            unsigned long long *hdr =
                (unsigned long long *)(ex.ring + (size_t)(ex_k % (unsigned long long)ex.slots) * ex.stride);
            asm volatile("st.release.sys.global.u64 [%0], %1;" ::"l"(hdr), "l"(ex_k + 1ull) : "memory");
            *ex.count = ex_k + 1ull;
        }
    }
    if (tid == 0) counters[ii] = 0u;
}

// The profiles a bead phase keeps (PhiTab), from a table's positions.
__global__ void k_phi(const Inst *__restrict__ insts, const int4 *__restrict__ blist, const BeadTab tab0,
                      const BeadTab tab1, const PhiTab phi0, const PhiTab phi1, int gparity) {
    const int4 br = blist ? blist[blockIdx.x] : make_int4(0, blockIdx.x, 0, gridDim.x);
    const Inst &I = insts[br.x >> 1];
    const bool one = gparity ^ (br.x & 1);
    const BeadTab &tab = one ? tab0 : tab1;
    const PhiTab &pt = one ? phi0 : phi1;
    if (I.phi_cap == 0) return;
    const int b = br.y;
    const double rx = tab.Rx[b], ry = tab.Ry[b];
    const float xh = (float)rx, yh = (float)ry;
    const bool far = far_off(xh, yh);
    Support bx;
    support_axis(I, 0, xh, (float)(rx - (double)xh), far, rx, ry, bx.lo[0], bx.n[0], bx.rel[0]);
    support_axis(I, 1, yh, (float)(ry - (double)yh), far, rx, ry, bx.lo[1], bx.n[1], bx.rel[1]);
    const int ncell = bx.n[0] * bx.n[1];
    if (threadIdx.x == 0) pt.box[b] = make_int4(bx.lo[0], bx.lo[1], bx.n[0], bx.n[1]);
    double *phi = pt.phi + I.phi_off + (b - br.z) * I.phi_cap;
    for (int c = threadIdx.x; c < ncell && c < I.phi_cap; c += blockDim.x) {
        int i = bx.lo[0] + c % bx.n[0], j = bx.lo[1] + c / bx.n[0];
        i = (i >= I.nx) ? i - I.nx : i;
        j = (j >= I.ny) ? j - I.ny : j;
        phi[c] = phi_f64(I, i + 0.5, j + 0.5, rx, ry);
    }
}

}  // namespace

namespace {

// SMs of the current device (cached per device; 0 if unknown).
int sm_count() {
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
        cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

template <class S>
cudaError_t launch_beads_t(cudaLaunchConfig_t &cfg, int threads, bool team, const Inst *inst_d, const int4 *blist,
                           const void *pool, const BeadTab tab[2], const PhiTab phi[2], unsigned *mask_write,
                           int gparity, int advance, int wait_first, unsigned *counters, BeadExport ex,
                           unsigned *status) {
    constexpr bool kF64 = std::is_same<S, double>::value;
    cfg.blockDim = dim3(threads);
    typename PhiArg<S>::type p0, p1;
    if constexpr (kF64) p0 = phi[0], p1 = phi[1];
    auto *k = k_beads<S, kBeadThreads, false>;
    if constexpr (!kF64) {
        if (threads == kBeadThreadsFew) k = team ? k_beads<S, kBeadThreadsFew, true> : k_beads<S, kBeadThreadsFew, false>;
        if (threads == kBeadThreadsMid) k = k_beads<S, kBeadThreadsMid, false>;
    }
    return cudaLaunchKernelEx(&cfg, k, inst_d, blist, (const S *)pool, tab[0], tab[1], p0, p1, mask_write, gparity,
                              advance, wait_first, counters, ex, status);
}

// Most beads of an instance that form a cluster on the current device: more
// than 8 CTAs are beyond the portable size, and need the device's leave.
int team_limit() {
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int most = cache[dev].load(std::memory_order_relaxed);
    if (most) return most;
    most = kTeamBeads;
    const void *k[] = {(const void *)k_beads<float, kBeadThreadsFew, true>,
                       (const void *)k_beads<__half, kBeadThreadsFew, true>};
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = kTeamBeads;
    a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kTeamBeads);
    cfg.blockDim = dim3(kBeadThreadsFew);
    cfg.attrs = a;
    cfg.numAttrs = 1;
    for (const void *f : k) {
        int n = 0;
        if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess || n < 1)
            most = 8;
    }
    (void)cudaGetLastError();
    cache[dev].store(most, std::memory_order_relaxed);
    return most;
}

}  // namespace

void prepare_bead_kernels() { (void)team_limit(); }

cudaError_t launch_beads(int precision, const Inst *inst_d, const int4 *blist, int nb_total, int each, int box, int ntiles,
                         const void *pool, const BeadTab tab[2], const PhiTab phi[2], unsigned *mask_write, int gparity, int advance,
                         unsigned *counters, int pdl, cudaStream_t st, BeadExport ex, unsigned *status) {
    if (nb_total <= 0) return cudaSuccess;
    // one CTA per bead: a grid capped at the resident CTAs (persistent) keeps
    // the bead CTAs on the SMs at once and leaves the sweep that follows
    // too few registers to start its unmarked tiles with (measured with
    // 256-thread CTAs: the batched step 8 % slower), so every bead gets its
    // own CTA; a list that fits on the SMs one bead per SM gets wider CTAs
    const int sms = sm_count();
    const bool few = nb_total <= sms;
    // FP64: an SM issues one FP64 warp instruction per 16 cycles, so a short
    // list's beads are split over as many SMs as there are, up to kBeadParts
    // CTAs a bead
    int parts = 1;
    if (precision == 0)
        while (2 * parts <= kBeadParts && 2 * parts * nb_total <= 2 * sms) parts *= 2;
    // A sweep of up to a few waves has room for the bead CTAs beside it: they
    // list their supports while it runs.  They enter a longer sweep's SMs
    // only as it drains; then the next sweep's release comes first.  us a
    // step, listing first / waiting first, FP32 (FP16): 2048 tiles 12.0 / 14.9
    // (12.4 / 15.4), 4096 13.5 / 16.3 (13.0 / 16.7), 8192 23.3 / 22.4 (22.2 /
    // 19.9 with one cell a thread, 16.6 / 17.9 with two), 16384 45.2 / 43.6
    // (31.2 / 29.1)
    const int wait_first = ntiles > kEarlyListTiles ? 1 : 0;
    // Every instance of the launch has `each` beads (0: not all the same): its
    // CTAs form a cluster where there is room beside the sweep for one
    const bool team = precision != 0 && few && !wait_first && advance && !ex.ring && each >= 1 && each <= team_limit();
    // Threads a CTA, us a step.  A short list without clusters beside a sweep of
    // up to a few waves, 512 against 256, FP32 (FP16): boxes of up to 512 cells,
    // two rounds of 256 threads (kWideBox; phi_cells has four more an axis), at
    // 242 tiles and 3 x 9 beads, box of 225 cells 10.07 / 9.57 (11.34 / 10.90),
    // 484 10.55 / 10.20 (11.61 / 11.36); 600 tiles 10.22 / 9.71 (11.69 / 11.70),
    // 10.74 / 10.33 (11.98 / 11.92); 1024 tiles 10.46 / 10.40 (12.10 / 11.77),
    // 10.94 / 10.94 (12.36 / 11.80); 3616 tiles 11.55 / 11.63 (12.50 / 12.42),
    // 12.0 / 12.38 (12.87 / 12.84): past two tiles an SM the gain is not there
    // in every storage.  Larger boxes, 242 tiles: 576 cells 9.88 / 10.39, 625
    // 10.67 / 10.92 (11.46 / 11.33), 784 10.2 / 11.2, 1296 12.3 / 14.7; 1024
    // tiles, 625 cells 10.77 / 11.66 (12.06 / 12.30).  Clusters: 160 x 160 and
    // one bead of a 37 x 37 box 9.2 / 10.9.  Beside a long sweep the narrower
    // CTAs leave it more room: 4096 x 1024 FP16 27.05 / 26.64, FP32 43.86 /
    // 43.57 (128 threads: 26.89 and 44.85).  FP64, bound by its instructions,
    // 512 / 256 / 128: 80 x 40 27.8 / 26.5 / 26.1, 200 x 100 256 / 128 26.2 /
    // 25.6, 4096 x 1024 498 / 486.1 / 485.4.  Long lists: 128 (six CTAs an SM).
    int threads = kBeadThreads;
    if (precision != 0 && few) {
        const bool narrow = wait_first || (!team && box <= kWideBox && ntiles <= 2 * sms);
        threads = narrow ? kBeadThreadsMid : kBeadThreadsFew;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb_total * parts);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (parts > 1 || team) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = team ? each : parts;
        attr[na].val.clusterDim.y = 1;
        attr[na++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    switch (precision) {
        case 0:
            return launch_beads_t<double>(cfg, threads, team, inst_d, blist, pool, tab, phi, mask_write, gparity, advance,
                                          wait_first, counters, ex, status);
        case 1:
            return launch_beads_t<float>(cfg, threads, team, inst_d, blist, pool, tab, phi, mask_write, gparity, advance,
                                         wait_first, counters, ex, status);
        case 2:
            return launch_beads_t<__half>(cfg, threads, team, inst_d, blist, pool, tab, phi, mask_write, gparity, advance,
                                          wait_first, counters, ex, status);
    }
    return cudaErrorInvalidValue;
}

int phi_cells(const Inst &I) {
    // support_axis: at most 2 rcut + 5 cells an axis, and two for its FP32 rounding
    const double n = 2.0 * I.rcut + 8.0;
    const int64_t w = n < I.nx ? (int64_t)n : I.nx, h = n < I.ny ? (int64_t)n : I.ny;
    return (int)(w * h);
}

cudaError_t launch_phi(const Inst *insts, const int4 *blist, int nb_total, const BeadTab tab[2], const PhiTab phi[2],
                       int gparity, cudaStream_t st) {
    if (nb_total <= 0) return cudaSuccess;
    k_phi<<<nb_total, 256, 0, st>>>(insts, blist, tab[0], tab[1], phi[0], phi[1], gparity);
    return cudaGetLastError();
}

}  // namespace fpd
