// Tree walk + node->ray mapping + far-to-near sweep, one CTA per target.
//
// A persistent grid takes targets (cells) from a job list: a job is one
// built tree and a range or list of its cells, so one launch can serve
// several independent problems.
// Walk (Sec. 2.3-2.4): the CTA keeps the opened nodes in a ring buffer in
// shared memory.  Each step takes up to NT/8 of them and evaluates their NT
// children at once, one child per thread: a child that contains the target,
// or fails the BH MAC (h/d < theta_lim), the IF MAC (nodes holding an
// ionisation front: h/d < theta_IF) or the Src MAC (emitting nodes:
// h/d < theta_src), is pushed as opened; the others are accepted and listed.
// On an AMR tree a node flagged as a cell is never opened.
// In the FP32 forms the distances come from FP32 records, and every opening
// decision and every discontinuous choice of the radial spreading (beyond
// L_ray or not, beyond the last point or not, a kernel support that is empty
// or holds one point) that FP32 cannot settle within a certified bound on
// its distance error is re-taken in FP64 from an FP64 copy of the tree: the
// accepted nodes are those of the FP64 form, bit for bit.
// Map (Sec. 2.3, App. A): the warps spread the listed nodes, 32 at a time,
// over the rays their table entry lists (angular weights) and the
// evaluation points their radial kernel reaches (W_p or W_g for the
// recombination rate alpha and the energy e; W_f,3 or another flux kernel
// for the emission eps), with shared-memory atomics into the ray bins: FP64
// adds in the FP64 form, exact 64-bit fixed point in the FP32 forms.
// Sweep (Sec. 2.5, Eq. 12-17): each ray is swept far to near (FP64 and
// FP32 + FP64-sweep forms: FP64 arithmetic, a lane per emitting point while a
// target has few, else a lane pair per ray, a warp per ray with a lone source;
// FP32 + double-FP32-sweep form: FP32 losses, double-FP32 budgets, a lane per
// source or a pair per ray) and the CTA sums the rays (Eq. 18).
// Variants: CTAs of 128, 256 or 512 threads by the room that the bins leave
// (pick_cta), a dump mode keeping the raw bins and accepted ids, a
// column-density mode without radial points, and a separate instantiation for
// non-default kernels and boundaries.
#include <algorithm>
#include <mutex>
#include <vector>

#include "tr_internal.cuh"

namespace tr {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// MODE 0: FP64 form; 1: FP32 walk + FP64 sweep; 2: FP32 walk + double-FP32 sweep
template <int MODE> struct Prec;
template <> struct Prec<0> { using real = double; using Node = NodeF64; };
template <> struct Prec<1> { using real = float; using Node = NodeF32; };
template <> struct Prec<2> { using real = float; using Node = NodeF32; };

constexpr float U32 = 5.9604645e-8f;        // 2^-24, the unit roundoff of FP32

struct WalkArgs {
    const void* nodes;
    const NodeF64* nodes64;                 // FP32 forms: the FP64 tree (exact re-decisions)
    const float* kappa;                     // FP32 forms: |cm32 - cm64| <= kappa x edge
    int N, L, nr, npix, eta, nside, use_e;
    double th_lim2, th_if2, th_src2, lray;
    double r_coef;                          // r_i = i^2 r_coef cells, r_coef = 1 / (2 eta^2) (Eq. 4)
    float r_coeff;                          // the same (a power of two: exact in FP32)
    float th_lim2f, th_if2f, th_src2f, lrayf;
    const uint32_t* toff;
    const uint32_t* tent;
    const uint2* hdr;
    const double* r;
    const float* rf;
    const double* inv_r2;
    const double* inv_vol;
    const float* inv_volf;
    const double* HT;                       // [j][i] lone-source loss per raw recombination deposit
    const double* ID2;
    const double* GI;
    const float* Gf;
    const float* ID2f;
    const float* GIf;
    const int64_t* targets;                 // NULL: cells first .. first+n_targets-1 in walk order
    int64_t first;
    const uint8_t* flags;                   // AMR tree: node topology (NULL: uniform grid)
    const int4* blk;                        // AMR tree: per block {cell level, x, y, z}
    const uint32_t* blk_order;              // AMR tree: blocks in walk order
    int64_t n_cells;                        // valid target indices are [0, n_cells)
    int kern_a, kern_e;                     // tr_kernel (alpha, e) and tr_eps_kernel (eps)
    int bc;                                 // tr_bc of the walk
    double* cd_out;                         // column-density maps: [target][N_PIX], cm^-2
    double cd_conv;                         // n_H cells -> cm^-2 (the cell edge dx)
    double cd_omega;                        // 4 pi / N_PIX
    int64_t n_targets;
    double Fconv, Econv;                    // scaled flux -> CGS flux / energy density
    double* F;
    double* E;
    uint8_t* ion;
    double* bins_out;
    int32_t* ids_out;
    int32_t* counts_out;
    double* eps_self_out;
    float* scales_out;                      // dump: the fixed-point units of the FP32 form
    const float* scales_in;                 // stored sweep: the same, read back
    int acc_cap;
    int32_t* status;
    unsigned long long* stats;
};

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// GB300's FP64: each of an SM's four schedulers has a unit that takes 64 cycles
// per warp instruction, however many lanes it has, with no overlap (measured:
// 65 cycles per FMA for one warp, dependent or not; 16 per SM with four warps).
// So FP64 work is packed onto few warps, those warps lie on different
// schedulers from one CTA of an SM to the next, and conversions and
// comparisons go to the integer units.

// The nearest float towards zero of a double in the float range (bounds only).
__device__ __forceinline__ float narrow(double a) {
    return __uint_as_float(((uint32_t)__double2hiint(a) - 0x38000000u) << 3 | (uint32_t)__double2loint(a) >> 29);
}

// Comparisons of non-negative doubles: their bit patterns order like them.
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool nonzero(double x) { return (__double2hiint(x) | __double2loint(x)) != 0; }   // (or -0)
__device__ __forceinline__ bool less(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }

// W_p of App. A (Eq. A2), outer branch rebuilt from the constraints printed
// with it: W_p2(x) = (x - sqrt3/2)^2 (a2 x + 2A(2 + sqrt3) - a2/2).
template <typename T>
__device__ __forceinline__ T wp_kernel(T x) {
    const T a1 = T(1.21), a2 = T(-6.35), A = T(4.08), M = T(1.184);
    const T s3h = T(0.86602540378443864676);
    const T c2 = T(2.0) * A * (T(2.0) + T(1.73205080756887729353)) - T(0.5) * a2;
    if constexpr (sizeof(T) == 8) {          // FP64: evaluate only the branch needed
        if (x < T(0.5)) return M + x * x * (a1 * x - (T(0.5) * a1 + T(4.0) * (M - A)));
        if (x < s3h) { T t = x - s3h; return t * t * (a2 * x + c2); }
        return T(0);
    } else {                                 // FP32: both branches and a select (lanes of a warp
        const T inner = M + x * x * (a1 * x - (T(0.5) * a1 + T(4.0) * (M - A)));   // sit on either side)
        const T t = x - s3h;
        const T outer = t * t * (a2 * x + c2);
        return x < T(0.5) ? inner : (x < s3h ? outer : T(0));
    }
}

// W_p in FP64 for lanes on either side of its branches: both as k0 + u^2 (k1 +
// k2 u), u = x or x - sqrt3/2, the constants picked by integer selects.  Four
// FP64 instructions instead of seven and two comparisons.
__device__ __forceinline__ double wp_select(double x) {
    constexpr double a1 = 1.21, a2 = -6.35, A = 4.08, M = 1.184, s3h = 0.86602540378443864676;
    constexpr double c1 = 0.5 * a1 + 4.0 * (M - A), c2 = 2.0 * A * (2.0 + 1.73205080756887729353) - 0.5 * a2;
    const bool in = less(x, 0.5);
    const double u = x - (in ? 0.0 : s3h);
    const double w = fma(u * u, fma(in ? a1 : a2, u, in ? -c1 : c2 + a2 * s3h), in ? M : 0.0);
    return less(x, s3h) ? w : 0.0;
}

// W_g of App. A (Eq. A1): exp(-x^2), truncated at sqrt3/2.
constexpr double S3H_D = 0.86602540378443864676;

template <typename T>
__device__ __forceinline__ T wg_kernel(T x) {
    return x < T(S3H_D) ? exp(-x * x) : T(0);
}

// The smoothing kernel of alpha and e at distance `dist` from the node:
// W_p(dist / h) with hpar = 1/h, or W_g(dist / h) with hpar = h (a true
// division, since W_g jumps at its truncation and the argument must round
// as the definition's quotient does).
template <typename T>
__device__ __forceinline__ T radial_w(T dist, T hpar, int gauss) {
    return gauss ? wg_kernel<T>(dist / hpar) : wp_kernel<T>(dist * hpar);
}

// Stack entry standing for "evaluate the root node" (real entries hold a
// level <= 9 in their top 5 bits, so this value never occurs as one).
constexpr uint32_t ROOT_EVAL = 0xffffffffu;

// One axis of the node copy the boundary condition puts next to the target
// (Sec. 2.8): g2, t2 = twice the node's and the target's centre (finest
// cells).  Corner of symmetry, axis mirrored: the node seen from the
// mirrored target.  Periodic: the nearest copy, offset wrapped into [-N, N)
// half cells.
template <typename T>
__device__ __forceinline__ void bc_frame(int bc, int mirrored, int N, int g2, int t2, T p, int& o, T& q) {
    if (bc == TR_BC_CORNER && mirrored) { o = -(g2 + t2); q = -p; return; }
    o = g2 - t2;
    q = p;
    if (bc == TR_BC_PERIODIC) {
        if (o >= N) { o -= 2 * N; q += (T)N; }
        else if (o < -N) { o += 2 * N; q -= (T)N; }
    }
}

// Bin of face coordinate x / A (|x| < A or, on a tie, the last bin): floor(16
// |x| / A) from one approximate reciprocal rA of A.  (16 |x| + 1/2) / A lies
// at least 1 / (2A) >= 2.4e-4 from an integer (A < 2048) and the product is
// off by less than 1e-5, so the floor is exact without an integer division.
__device__ __forceinline__ int face_bin(int x, float rA) {
    const int q = min((int)(fmaf((float)abs(x), (float)TQH, 0.5f) * rA), TQH - 1);
    return x == 0 ? TQH : (x > 0 ? TQH + 1 + q : TQH - 1 - q);
}

// Table key of a node from the integer offset o = 2 (node centre - target
// centre) in half cells and the node edge s in cells: a face key when one
// axis has the largest |o|, an edge key when two tie for it, a corner key
// when all three do.  psi bin = floor(64 s / |o|), at most TB - 1: FP32 gives
// it to 3e-5, so the exact integer comparison is made only within 1e-4 of an
// integer (a bin in ten thousand).
__device__ __forceinline__ int table_key(int ox, int oy, int oz, int s) {
    const int ax = abs(ox), ay = abs(oy), az = abs(oz);
    const int A = max(ax, max(ay, az));
    const int o2 = ox * ox + oy * oy + oz * oz;              // < 3 x 2048^2: exact, also as a float
    const float q = 64.f * (float)s * rsqrtf((float)o2);
    int pb = (int)fminf(q, (float)(TB - 1));
    if (q < (float)TB && fabsf(q - rintf(q)) < 1e-4f) {
        const long long lim = 64LL * s, lim2 = lim * lim;
        if ((long long)pb * pb * o2 > lim2) --pb;
        else if ((long long)(pb + 1) * (pb + 1) * o2 <= lim2) ++pb;
        pb = min(pb, TB - 1);
    }
    const float rA = __fdividef(1.f, (float)A);
    const bool tx = ax == A, ty = ay == A, tz = az == A;
    const int ntie = (int)tx + (int)ty + (int)tz;
    if (ntie == 1) {
        const int ob = tx ? oy : ox, oc = tz ? oy : oz, oa = tx ? ox : (ty ? oy : oz);
        const int face = (tx ? 0 : (ty ? 2 : 4)) + (oa < 0 ? 1 : 0);
        return ((face * TQ + face_bin(ob, rA)) * TQ + face_bin(oc, rA)) * TB + pb;
    }
    if (ntie == 2) {                         // edge of the tied axes a < b, the third axis c binned
        const int c = !tx ? 0 : (!ty ? 1 : 2);
        const int pair = c == 2 ? 0 : (c == 1 ? 1 : 2);
        const int oa = c == 0 ? oy : ox, ob = c == 2 ? oy : oz, oc = c == 0 ? ox : (c == 1 ? oy : oz);
        const int edge = 4 * pair + 2 * (oa < 0) + (ob < 0);
        return NFACEKEYS + (edge * TQ + face_bin(oc, rA)) * TB + pb;
    }
    const int corner = (ox < 0) + 2 * (oy < 0) + 4 * (oz < 0);
    return NFACEKEYS + NEDGEKEYS + corner * TB + pb;
}

// Ray bins.  FP64 form: one double per bin, atomic FP64 adds.  FP32 form: the
// FP32 addends are accumulated exactly in 64-bit fixed point, kept as two
// 32-bit words (low word, high word) updated by two integer atomics with the
// carry of the low word propagated: an order-independent sum whose only
// rounding is that of each FP32 addend.  The fixed-point unit is a power of
// two chosen from the root node's total, so that no bin can exceed 2^62.
struct Scales { float a, eps, e; };          // fixed-point units per quantity (FP32 form)

__device__ __forceinline__ float fixed_scale(float total) {
    int ex = 0;
    frexpf(total > 0.f ? total : 1.f, &ex);   // total < 2^ex
    return ldexpf(1.0f, min(62 - ex, 126));
}

// A bin times f: FP32 forms, f holds the reciprocal of the unit (a power of two).
template <int MODE>
__device__ __forceinline__ double bin_value(const double* slot, double f) {
    if (MODE == 0) return *slot * f;
    const uint2 v = *reinterpret_cast<const uint2*>(slot);
    // 2^84 + high x 2^32 and 2^52 + low, without a conversion
    const double h = __hiloint2double(0x45300000, (int)v.y), l = __hiloint2double(0x43300000, (int)v.x);
    return ((h - 19342813118337666422669312.0) + l) * f;
}

template <int MODE>
__device__ __forceinline__ float bin_value_f(const double* slot, float inv_scale) {
    const uint2 v = *reinterpret_cast<const uint2*>(slot);
    return ((float)v.y * 4294967296.0f + (float)v.x) * inv_scale;
}

template <int MODE>
__device__ __forceinline__ bool bin_nonzero(const double* slot) {
    if (MODE == 0) return *slot > 0.0;
    const uint2 v = *reinterpret_cast<const uint2*>(slot);
    return (v.x | v.y) != 0u;
}

// FP32 forms: add v >= +0 (in units of the bin, below 2^62; the caller sees to
// it: the sign bit would be read as part of the exponent, so that -0 would add
// 2^33 units), rounded down to an integer, to a bin.  Integer placement of the
// significand rather than two float-to-integer conversions: those share a pipe
// of 16 lanes per SM and clock (turbulent128, double-FP32 form: 232 -> 226 ms;
// the unconditional second atomic 226 -> 217 ms).
__device__ __forceinline__ void bin_add_units(double* slot, float v) {
    unsigned* w = reinterpret_cast<unsigned*>(slot);
    // the 24-bit significand placed in 64 bits by one widening multiply
    const uint32_t b = __float_as_uint(v);
    const int t = (int)(b >> 23) - 126;                       // v in [2^(t-1), 2^t)
    const uint64_t p = (uint64_t)((b << 8) | 0x80000000u) * (1u << (t & 31));
    const uint32_t pl = (uint32_t)p, ph = (uint32_t)(p >> 32);
    const uint32_t lo = t >= 32 ? pl : (t > 0 ? ph : 0u), hi = t >= 32 ? ph : 0u;
    const unsigned old = atomicAdd(w, lo);
    unsigned h;
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 %0, %3, 0;\n\t}" : "=r"(h) : "r"(old), "r"(lo), "r"(hi));
    atomicAdd(w + 1, h);                                      // (a branch around zero costs more)
}

template <int MODE>
__device__ __forceinline__ void bin_atomic_add(double* slot, typename Prec<MODE>::real x, float scale) {
    if constexpr (MODE == 0) atomicAdd(slot, (double)x);
    else if ((float)x > 0.f) bin_add_units(slot, (float)x * scale);   // exact: scale is a power of two
}

template <int MODE>
__device__ __forceinline__ void load_node(const void* nodes, int64_t id, typename Prec<MODE>::real* cm,
                                          typename Prec<MODE>::real& m, typename Prec<MODE>::real* q,
                                          typename Prec<MODE>::real& mion) {
    if (MODE == 0) {
        const double2* p = reinterpret_cast<const double2*>((const NodeF64*)nodes + id);
        const double2 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3);
        cm[0] = a.x; cm[1] = a.y; cm[2] = b.x; m = b.y;
        q[0] = c.x; q[1] = c.y; q[2] = d.x; mion = d.y;
    } else {
        const float4* p = reinterpret_cast<const float4*>((const NodeF32*)nodes + id);
        const float4 a = __ldg(p), b = __ldg(p + 1);
        cm[0] = a.x; cm[1] = a.y; cm[2] = a.z; m = a.w;
        q[0] = b.x; q[1] = b.y; q[2] = b.z; mion = b.w;
    }
}

// Opening decision of a non-leaf node that does not contain the target (an
// infinite angle always accepts, so its products are not formed).
__device__ __forceinline__ bool must_open(double h2, double d2, double m, double mion, double eps,
                                          const WalkArgs& a) {
    if (!less(h2, __dmul_rn(a.th_lim2, d2))) return true;
    if (isfinite(a.th_if2f) && __dmul_rn(DELTA_IF, m) < mion && mion < __dmul_rn(1.0 - DELTA_IF, m) &&
        !less(h2, __dmul_rn(a.th_if2, d2)))
        return true;
    return isfinite(a.th_src2f) && positive(eps) && !less(h2, __dmul_rn(a.th_src2, d2));
}
// The same decision taken in FP64 with the node's IF flag given (FP32 forms,
// when FP32 cannot settle it).
__device__ __forceinline__ bool must_open_exact(double h2, double d2, bool is_if, bool has_eps, const WalkArgs& a) {
    const bool acc_lim = h2 < __dmul_rn(a.th_lim2, d2);
    const bool acc_if = !is_if || (h2 < __dmul_rn(a.th_if2, d2));
    const bool acc_src = !has_eps || (h2 < __dmul_rn(a.th_src2, d2));
    return !(acc_lim && acc_if && acc_src);
}

// Bound on |d2 - d2_64| for an FP32 squared distance d2 whose per-axis
// displacement carries an error of at most E from the stored centre of mass
// (plus the rounding of the displacement, the squares and the sums): with
// e_a <= E + u d per axis, |sum dx^2 - sum dx64^2| <= 2 sqrt3 d e + 3 e^2,
// plus 3.1 u d2 of rounding; a factor 2 of margin on top.
__device__ __forceinline__ float d2_err_bound(float d2, float E) {
    const float d = d2 * rsqrtf(d2) * 1.000001f;
    const float e = E + 1.01f * U32 * d;
    return 2.f * (3.4641017f * d * e + 3.f * e * e + 3.1f * U32 * d2);
}

// One criterion h2 < t2 d2_64 with d2_64 in [lo, hi]: 1 surely true, 0 surely
// false, -1 undecided (lo and hi carry the roundings of t2 and the product).
__device__ __forceinline__ int mac_tri(float h2, float t2, float lo, float hi) {
    if (h2 < t2 * lo) return 1;
    if (h2 >= t2 * hi) return 0;
    return -1;
}

// Opening decision of the FP32 forms: 1 open, 0 accept, -1 undecided within
// the error bound B of d2 (then taken by must_open_exact on FP64 data).
__device__ __forceinline__ int mac_f32(float h2, float d2, float B, bool is_if, bool has_eps, const WalkArgs& a) {
    const float lo = fmaxf(d2 - B, 0.f) * (1.f - 8.f * U32);
    const float hi = (d2 + B) * (1.f + 8.f * U32);
    int r = mac_tri(h2, a.th_lim2f, lo, hi);
    if (r == 0) return 1;
    bool und = r < 0;
    if (is_if) { r = mac_tri(h2, a.th_if2f, lo, hi); if (r == 0) return 1; und |= r < 0; }
    if (has_eps) { r = mac_tri(h2, a.th_src2f, lo, hi); if (r == 0) return 1; und |= r < 0; }
    return und ? -1 : 0;
}

__device__ __forceinline__ double dist2(double tx, double ty, double tz, const double* cm) {
    const double dx = __dsub_rn(tx, cm[0]), dy = __dsub_rn(ty, cm[1]), dz = __dsub_rn(tz, cm[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}
// FP32 forms: the squared distance of node nid from the target centre (tx,
// ty, tz) in FP64 from the FP64 tree, exactly as the FP64 form computes it.
__device__ __forceinline__ double exact_d2(const WalkArgs& a, int64_t nid, float tx, float ty, float tz) {
    const double2 c01 = __ldg(reinterpret_cast<const double2*>(a.nodes64 + nid));
    const double cm[3] = {c01.x, c01.y, __ldg(&a.nodes64[nid].cmz)};
    return dist2((double)tx, (double)ty, (double)tz, cm);
}

// Radial spread of one accepted node (App. A), prepared by one lane: the
// points lo .. lo+npts-1 and their weights.  The weights are the values that
// the lane keeps in its column of the warp's NodeBatch, times b; a support
// of more than MAXW points is evaluated again for each ray instead (`lng`:
// column entries 0 and 1 then hold d and the kernel's size argument).
// Kernel values kept per node.  A longer support, met by the few nodes with
// edges of 32 cells and more, costs its evaluation again per ray.
// FP64: 12, evaluating again costs more.  FP32: 7, so that a 128-thread CTA
// takes 9.7 KB beside its ray bins and as many targets fit an SM as should: five
// at 33 KB of bins (N_PIX 48, N_R 43; with 12 values only four: 225 -> 253 ms),
// four at 45 KB (N_R 59; with 8 only three, by 256 bytes: a 256^3 grid with 100
// sources 406 -> 329 ms per 2^20 targets, headline form).  8 where six CTAs fit
// (the bins leave room), and for the other radial kernels, whose evaluation is
// an exponential and a division (W_g headline walk of 32^3: 1.82 -> 1.72 ms).  6
// in the slim 512-thread CTA (see pick_cta).
template <int MODE, int NT, int CTAS, bool VAR, bool SLIM>
constexpr int MAXW = MODE == 0 ? 12 : (SLIM ? 6 : (NT == 128 && (CTAS == 6 || VAR) ? 8 : 7));

template <int MODE>
struct RadialSpread {
    typename Prec<MODE>::real b;
    int lo, npts;
    bool lng;
};

// The accepted nodes that one warp spreads together (32 at most), in shared
// memory: kernel values in a column per set-up lane (conflict-free for lanes
// that read different nodes at the same point), the rest by the node's rank
// among the nodes with work.
template <int MODE, int W>
struct __align__(16) NodeBatch {
    using real = typename Prec<MODE>::real;
    real w[W][32];
    uint2 key[32];                          // {first table entry less first (node, ray) pair, points packed}
    real a[32], b[32];                      // alpha, weight factor (FP64 form: alpha x b / TW, -)
    real e[32];                             // e (FP64 form: e x b / TW)
    real eps[32], w1[32];                   // eps and the share of its second point (W_f,3)
};
// packing of a node's points: lo (7 bits), npts (8), set-up lane (5), first
// point of eps (7), flags
constexpr uint32_t PK_EPS = 1u << 27, PK_LONG = 1u << 28;

// r_i of Eq. 4: in FP32 from its index, i^2 times a power of two (exact, no
// load); in FP64 from the table (an FP64 multiply costs more than the load)
template <typename T>
__device__ __forceinline__ T radius_at(int i, T coef, const double* tab) {
    if constexpr (sizeof(T) == 8) return __ldg(tab + i);
    else return (T)(i * i) * coef;
}

// W_p normalisation of an accepted node in the FP32 forms: the support of the
// kernel on the evaluation points and 1/S.  dtol bounds the error of d; returns
// true when a discontinuous choice -- d beyond the last point or
// not, or a support that is empty or holds only points within rounding of
// its edge (the normalisation then jumps between one point and the linear
// split) -- is not settled in FP32; radial_setup_exact then takes it in FP64.
template <int MODE, int W>
__device__ __forceinline__ bool radial_setup(const WalkArgs& a, RadialSpread<MODE>& n, float d, int s, float* wcol, int gauss,
                                             float dtol) {
    const int nr = a.nr;
    const float rc = a.r_coeff;
    n.b = 1.f; n.lng = false;
    const float rlast = radius_at<float>(nr - 1, rc, a.r);
    if (d >= rlast) {
        n.lo = nr - 1; n.npts = 1; wcol[0] = 1.f;
        return d - dtol < rlast;
    }
    if (d + dtol >= rlast) return true;
    const float h = (float)s, inv_h = 1.f / h;
    const float hpar = gauss ? h : inv_h;
    const float reach = 0.8661f * h + dtol;
    const float dlo = d > reach ? d - reach : 0.f;
    // floor / ceil of the support's index bounds (i = eta sqrt(2 r), Eq. 4),
    // from approximate roots and a margin above their error: it only widens the
    // range by a point whose weight is zero
    const float el = 2.f * dlo, eh = 2.f * (d + reach);
    const int lo = max((int)((float)a.eta * (el * rsqrtf(fmaxf(el, 1e-30f))) - 1e-3f), 0);
    const int hi = min((int)((float)a.eta * (eh * rsqrtf(eh)) + 1.001f), nr - 1);
    float S = 0.f;
    int cnt = 0, last = lo - 1;
    float near = 1e30f;                     // the closest point
    float* col = wcol;
    float fi = (float)lo;
    for (int i = lo; i <= hi; ++i, fi += 1.f) {
        const float dist = fabs((fi * fi) * rc - d);
        const float w = radial_w<float>(dist, hpar, gauss);
        near = fmin(near, dist);
        if (w > 0.f) {                      // the support is one run of points
            S += w;
            last = i;
            if (cnt < W) *col = w;
            col += 32;
            ++cnt;
        }
    }
    // a point whose kernel argument lies within xtol of sqrt3/2 may fall on the
    // other side of the support's edge in FP64; that matters when no point is
    // surely inside, i.e. when the closest one is not
    const float xtol = 2.f * (dtol + U32 * (2.f * d + reach)) * inv_h + 4.f * U32;
    const float x = near * inv_h - (float)S3H_D;
    if (!(x < -xtol) && x <= xtol) return true;
    if (cnt > 0) {
        n.lo = last - cnt + 1; n.npts = cnt; n.b = 1.f / S;
        if (cnt > W) { n.lng = true; wcol[0] = d; wcol[32] = hpar; }
        return false;
    }
    int i = min(max((int)floorf((float)a.eta * sqrtf(2.f * d)), 0), nr - 2);   // a guess, corrected below
    while (i + 1 < nr - 1 && radius_at<float>(i + 1, rc, a.r) <= d) ++i;
    while (i > 0 && radius_at<float>(i, rc, a.r) > d) --i;
    const float ra = radius_at<float>(i, rc, a.r), rb = radius_at<float>(i + 1, rc, a.r);
    n.lo = i; n.npts = 2;
    wcol[0] = (rb - d) / (rb - ra);
    wcol[32] = (d - ra) / (rb - ra);
    return false;
}

// The other eps kernels (App. A.3), in FP64 whatever the form: emitting
// nodes are few.  The weights of points lo .. lo+n-1 are p0, p1 (two
// points), a + b k (generalised W_f,3, p0 = a, p1 = b) or a smoothing
// kernel over 1/S (p0).
struct EpsSpread {
    int lo, n, kind;                        // kind 0 two points, 1 linear, 2 W_p, 3 W_g
    double p0, p1, d, h;
};

__device__ __forceinline__ int bracket_d(const double* r, int nr, int eta, double d) {
    int i = min(max((int)floor((double)eta * sqrt(2.0 * d)), 0), nr - 2);
    while (i + 1 < nr - 1 && r[i + 1] <= d) ++i;
    while (i > 0 && r[i] > d) --i;
    return i;
}

// The W_p normalisation in FP64, settled always.  Bound by the FP64 units, so six FP64
// instructions per point (the kernel's argument is one add, r_i / h being exact
// in FP32; four for the kernel, one for the sum) and none for the index bounds,
// comparisons and conversions: plain FP64 turbulent64 92 -> 70 ms, Stroemgren
// 32^3 7.5 -> 5.6 ms.
template <int W>
__device__ __forceinline__ void radial_setup64(const WalkArgs& a, RadialSpread<0>& n, double d, int s, double* wcol,
                                               int gauss) {
    const int nr = a.nr;
    n.b = 1.0; n.lng = false;
    if (!less(d, __ldg(a.r + nr - 1))) {
        n.lo = nr - 1; n.npts = 1; wcol[0] = 1.0;
        return;
    }
    // s is a power of two: 1 / h from its exponent
    const float hf = (float)s, inv_hf = __uint_as_float((254u << 23) - __float_as_uint(hf));
    const double h = widen_normal(hf), inv_h = widen_normal(inv_hf), hpar = gauss ? h : inv_h;
    const float df = narrow(d), reach = 0.8661f * hf, dlo = df > reach ? df - reach : 0.f;
    const float el = 2.f * dlo, eh = 2.f * (df + reach);
    const int lo = max((int)((float)a.eta * (el * rsqrtf(fmaxf(el, 1e-30f))) - 1e-3f), 0);
    const int hi = min((int)((float)a.eta * (eh * rsqrtf(eh)) + 1.001f), nr - 1);
    double S = 0.0;
    int cnt = 0, last = lo - 1;
    double* col = wcol;
    float fi = (float)lo;
    const double dh = d * inv_h;            // (exact)
    const float rch = a.r_coeff * inv_hf;
    for (int i = lo; i <= hi; ++i, fi += 1.f) {
        const double w = gauss ? radial_w<double>(fabs(__ldg(a.r + i) - d), hpar, 1)
                               : wp_select(fabs(widen_normal(fi * fi * rch) - dh));
        if (positive(w)) {                  // the support is one run of points
            S += w;
            last = i;
            if (cnt < W) *col = w;
            col += 32;
            ++cnt;
        }
    }
    if (cnt > 0) {
        n.lo = last - cnt + 1; n.npts = cnt; n.b = recip(S);
        if (cnt > W) { n.lng = true; wcol[0] = d; wcol[32] = hpar; }
        return;
    }
    const int i = bracket_d(a.r, nr, a.eta, d);
    const double ra = __ldg(a.r + i), rb = __ldg(a.r + i + 1);
    n.lo = i; n.npts = 2;
    wcol[0] = (rb - d) / (rb - ra);
    wcol[32] = (d - ra) / (rb - ra);
}

// FP32 forms: the radial set-up of an accepted node taken on its FP64
// distance d, when radial_setup could not settle it: a d within rounding of the
// last point, or a support that FP32 left open (at most two points, both at its
// edge, or none).  Few weights are stored explicitly: one point, two
// consecutive points, or the linear split between the points bracketing d.
template <int MODE>
__device__ void radial_setup_exact(const WalkArgs& a, RadialSpread<MODE>& n, double d, int s,
                                   typename Prec<MODE>::real* wcol, int gauss) {
    const int nr = a.nr;
    n.b = 1.f; n.lng = false;
    if (d >= __ldg(a.r + nr - 1)) {
        n.lo = nr - 1; n.npts = 1; wcol[0] = 1.f;
        return;
    }
    const double h = (double)s, inv_h = 1.0 / h, hpar = gauss ? h : inv_h;
    const double reach = 0.8661 * h;
    const int lo = max((int)floor((double)a.eta * sqrt(2.0 * fmax(d - reach, 0.0))) - 1, 0);
    const int hi = min((int)ceil((double)a.eta * sqrt(2.0 * (d + reach))) + 1, nr - 1);
    int first = -1, cnt = 0;
    double w0 = 0.0, w1 = 0.0, S = 0.0;
    for (int i = lo; i <= hi; ++i) {
        const double w = radial_w<double>(fabs(__ldg(a.r + i) - d), hpar, gauss);
        if (w > 0.0) {
            if (cnt == 0) { first = i; w0 = w; } else if (cnt == 1) { w1 = w; }
            S += w;
            ++cnt;
        }
    }
    if (cnt == 1) { n.lo = first; n.npts = 1; wcol[0] = 1.f; return; }
    if (cnt == 2) { n.lo = first; n.npts = 2; wcol[0] = (float)(w0 / S); wcol[32] = (float)(w1 / S); return; }
    if (cnt > 2) {                          // (only beside the last point) FP32 weights, evaluated per ray
        n.lo = first; n.npts = cnt; n.lng = true; n.b = (float)(1.0 / S);
        wcol[0] = (float)d; wcol[32] = (float)hpar;
        return;
    }
    const int i = bracket_d(a.r, nr, a.eta, d);
    const double ra = __ldg(a.r + i), rb = __ldg(a.r + i + 1);
    n.lo = i; n.npts = 2;
    wcol[0] = (float)((rb - d) / (rb - ra));
    wcol[32] = (float)((d - ra) / (rb - ra));
}

// two-point W_f,3: the sum and the flux at r = 0 exact
__device__ void eps_wf3(const double* r, int nr, int eta, double d, EpsSpread& s) {
    s.kind = 0;
    if (d >= r[nr - 1]) { s.lo = nr - 1; s.n = 1; s.p0 = 1.0; return; }
    const int i = bracket_d(r, nr, eta, d);
    if (i == 0) { s.lo = 1; s.n = 1; s.p0 = 1.0; return; }
    const double ri = r[i], rj = r[i + 1];
    const double ia = 1.0 / (ri * ri), ib = 1.0 / (rj * rj), it = 1.0 / (d * d);
    const double w1 = (ia - it) / (ia - ib);
    s.lo = i; s.n = 2; s.p0 = 1.0 - w1; s.p1 = w1;
}

__device__ void eps_setup(const WalkArgs& a, double d, double h, EpsSpread& s) {
    const double* r = a.r;
    const int nr = a.nr, eta = a.eta;
    s.d = d; s.h = h;
    if (a.kern_e == TR_EPS_WF1 || a.kern_e == TR_EPS_WF2) {
        // W_f,1: w_{i+1} / w_i = (d - r_i) / (r_{i+1} - d); W_f,2: the flux also
        // exact at r_{i-1}; both with the flux at r = 0 exact
        const int i = d >= r[nr - 1] ? nr - 1 : bracket_d(r, nr, eta, d);
        if (d >= r[nr - 1] || i == 0 || (a.kern_e == TR_EPS_WF2 && i < 2)) { eps_wf3(r, nr, eta, d, s); return; }
        const double ri = r[i], rj = r[i + 1];
        double w0, w1;
        if (a.kern_e == TR_EPS_WF1) {
            const double ratio = (d - ri) / (rj - d);
            w0 = 1.0 / ((d * d) * (1.0 / (ri * ri) + ratio / (rj * rj)));
            w1 = ratio * w0;
        } else {
            const double rm = r[i - 1];
            const double a11 = 1.0 / (ri * ri), a12 = 1.0 / (rj * rj), b1 = 1.0 / (d * d);
            const double a21 = 1.0 / ((ri - rm) * (ri - rm)), a22 = 1.0 / ((rj - rm) * (rj - rm));
            const double b2 = 1.0 / ((d - rm) * (d - rm));
            const double det = a11 * a22 - a12 * a21;
            w0 = (b1 * a22 - a12 * b2) / det;
            w1 = (a11 * b2 - a21 * b1) / det;
            if (!(w0 >= 0.0 && w1 >= 0.0)) { eps_wf3(r, nr, eta, d, s); return; }
        }
        s.kind = 0; s.lo = i; s.n = 2; s.p0 = w0; s.p1 = w1;
        return;
    }
    if (a.kern_e == TR_EPS_WF3N) {
        // Eq. A8-A10 over the points i >= 1 inside the support
        if (d >= r[nr - 1]) { eps_wf3(r, nr, eta, d, s); return; }
        int lo = -1, n = 0;
        for (int i = 1; i < nr; ++i)
            if (fabs(r[i] - d) < S3H_D * h) { if (lo < 0) lo = i; ++n; }
        if (n <= 2) { eps_wf3(r, nr, eta, d, s); return; }
        double A1 = 0.0, A2 = 0.0;
        for (int k = 0; k < n; ++k) {
            const double rk = r[lo + k];
            A1 += 1.0 / (rk * rk);
            A2 += (double)k / (rk * rk);
        }
        const double b = (1.0 / (d * d) - A1 / (double)n) / (A2 - (double)(n - 1) * A1 / 2.0);
        const double c = 1.0 / (double)n - b * (double)(n - 1) / 2.0;
        if (c < 0.0 || c + b * (double)(n - 1) < 0.0) { eps_wf3(r, nr, eta, d, s); return; }   // linear: ends suffice
        s.kind = 1; s.lo = lo; s.n = n; s.p0 = c; s.p1 = b;
        return;
    }
    // W_p or W_g normalised over the points, as for alpha
    const int gauss = a.kern_e == TR_EPS_WG;
    if (d >= r[nr - 1]) { s.kind = 0; s.lo = nr - 1; s.n = 1; s.p0 = 1.0; return; }
    double S = 0.0;
    int first = nr, last = -1;
    for (int i = 0; i < nr; ++i) {
        const double x = fabs(r[i] - d) / h;
        const double w = gauss ? wg_kernel<double>(x) : wp_kernel<double>(x);
        if (w > 0.0) { S += w; first = min(first, i); last = i; }
    }
    if (S > 0.0) { s.kind = gauss ? 3 : 2; s.lo = first; s.n = last - first + 1; s.p0 = 1.0 / S; return; }
    const int i = bracket_d(r, nr, eta, d);
    s.kind = 0; s.lo = i; s.n = 2;
    s.p0 = (r[i + 1] - d) / (r[i + 1] - r[i]);
    s.p1 = (d - r[i]) / (r[i + 1] - r[i]);
}

__device__ __forceinline__ double eps_weight(const EpsSpread& s, const double* r, int j) {
    if (s.kind == 0) return j == 0 ? s.p0 : s.p1;
    if (s.kind == 1) return s.p0 + s.p1 * (double)j;
    const double x = fabs(r[s.lo + j] - s.d) / s.h;
    return (s.kind == 3 ? wg_kernel<double>(x) : wp_kernel<double>(x)) * s.p0;
}

// eps deposit with a kernel other than the default.
template <int MODE>
__device__ __forceinline__ void deposit_eps_variant(const WalkArgs& a, double* bins_eps, uint32_t off, int ne, double d,
                                                 typename Prec<MODE>::real eps, float scale, int s_edge) {
    using real = typename Prec<MODE>::real;
    const int nr = a.nr;
    EpsSpread sp;
    eps_setup(a, d, (double)s_edge, sp);
    const real inv_m3v = real(1.0) / real(TW);
    for (int k = 0; k < ne; ++k) {
        const uint32_t en = __ldg(a.tent + off + k);
        const int b = (int)(en >> 16) * nr + sp.lo;
        const real wk = (real)(en & 0xffffu) * inv_m3v;
        for (int j = 0; j < sp.n; ++j) {
            const real w = (real)eps_weight(sp, a.r, j);
            if (w != real(0)) bin_atomic_add<MODE>(bins_eps + b + j, wk * w * eps, scale);
        }
    }
}

// The default eps kernel W_f,3 (App. A.3): two points r_i <= d < r_{i+1}
// keeping the sum and the flux at the target exact (a continuous function of
// d).  Returns i; the second point's share in w1, the first's is 1 - w1.
template <int MODE>
__device__ __forceinline__ int eps_split(const WalkArgs& a, typename Prec<MODE>::real d, typename Prec<MODE>::real& w1) {
    using real = typename Prec<MODE>::real;
    const int nr = a.nr;
    const real* r = (MODE == 0) ? reinterpret_cast<const real*>(a.r) : reinterpret_cast<const real*>(a.rf);
    w1 = real(1);
    if (d >= r[nr - 1]) return nr - 2;
    int i = min(max((int)floorf((float)a.eta * sqrtf(2.f * (float)d)), 0), nr - 2);   // a guess, corrected below
    while (i + 1 < nr - 1 && r[i + 1] <= d) ++i;
    while (i > 0 && r[i] > d) --i;
    if (i > 0) {
        const real ri = r[i], rj = r[i + 1];
        const real ia = real(1) / (ri * ri), ib = real(1) / (rj * rj), it = real(1) / (d * d);
        w1 = (ia - it) / (ia - ib);
    }
    return i;
}

// Recombination coefficient per unit volume at point i of a ray.  In the
// FP32 + FP64-sweep form the deposits are FP32, so the coefficient is formed
// in FP32 and widened; the photon budget (Phi_j, its losses and their
// clipping) is FP64.
// The widening takes the power of two of the bin's unit (unit_base), so that no
// FP32 value leaves the normal range.
__device__ __forceinline__ int unit_base(float scale) {      // of 1 / scale, scale a power of two
    return 0x38000000 + (127 - (int)(__float_as_uint(scale) >> 23)) * (1 << 20);
}
__device__ __forceinline__ float bin_units(const double* slot) {
    const uint2 v = *reinterpret_cast<const uint2*>(slot);
    return (float)v.y * 4294967296.0f + (float)v.x;
}
template <int MODE>
__device__ __forceinline__ double alpha_at(const WalkArgs& a, const double* ba, int i, int unit) {
    if (MODE == 0) return ba[i] * __ldg(a.inv_vol + i);
    return widen_scaled(bin_units(ba + i) * __ldg(a.inv_volf + i), unit);
}

// Flux at r = 0 of a ray with a lone source at jtop and no e, by a whole warp
// (lane 0 returns it): zeta_s = zeta_d = 1 on every segment and every R_ij >=
// 0, so that clipping once at the end equals clipping per segment (Eq. 13):
// Phi_0 = max(Phi_j - sum_i bin_i HT[j][i], 0).
template <int MODE>
__device__ __forceinline__ double lone_ray(const WalkArgs& a, const double* ba, const double* be, const Scales& sc, int jtop) {
    const int lane = threadIdx.x & 31;
    const int ia = unit_base(sc.a);
    const double* h = a.HT + (size_t)jtop * a.nr;
    double s0 = 0.0;
    for (int i = lane; i <= jtop; i += 32)
        s0 = fma(MODE == 0 ? ba[i] : widen_scaled(bin_units(ba + i), ia), __ldg(h + i), s0);
    s0 = warp_sum(s0);
    const double phi = bin_value<MODE>(be + jtop, (MODE == 0 ? 1.0 : 1.0 / (double)sc.eps) * (1.0 / (4.0 * PI_D))) - s0;
    return positive(phi) && lane == 0 ? phi * __ldg(a.inv_r2 + jtop) : 0.0;
}

// Readies one ray for the FP64 sweep, by a whole warp (a lane per segment, so
// that the FP64 units see one instruction for 32 segments): leaves in ba[i],
// i < jtop, the loss coefficient A_i = alpha_i + alpha_{i+1} of segment i (Eq.
// 14; G carries the 1/2).  With the energy density e, zeta_d = min(2, F_tot /
// e) (Eq. 17), so the loss per unit of F_j G_ij is A zeta_d / F_tot = min(2 A /
// F_tot, A / e): where e > 0 at the segment's far point, ba[i] holds 2 A and
// bee[i] the limit A / e (else infinity).
template <int MODE>
__device__ __forceinline__ void prepare_ray(const WalkArgs& a, double* ba, double* bee, const Scales& sc, int jtop) {
    const int lane = threadIdx.x & 31, ia = unit_base(sc.a), ie = unit_base(sc.e);
    for (int base = 0; base < jtop; base += 32) {
        const int i = base + lane;
        double A = 0.0, Q = 0.0;
        if (i < jtop) {
            A = alpha_at<MODE>(a, ba, i, ia) + alpha_at<MODE>(a, ba, i + 1, ia);
            if (bee) {
                const double ev = alpha_at<MODE>(a, bee, i + 1, ie);
                Q = __longlong_as_double(0x7ff0000000000000LL);
                if (positive(ev)) { Q = A * recip(ev); A = A + A; }
            }
        }
        __syncwarp();                                         // raw values read before they are replaced
        if (i < jtop) { ba[i] = A; if (bee) bee[i] = Q; }
        __syncwarp();
    }
}

__device__ __forceinline__ int farthest(uint64_t m0, uint64_t m1) {
    return m1 ? 127 - __clzll((long long)m1) : (m0 ? 63 - __clzll((long long)m0) : 0);
}

// min(cf, limit): both >= 0, so their bit patterns compare like them.
__device__ __forceinline__ double loss_coef(double cf, const double* bee, int i) {
    if (!bee) return cf;
    const long long x = __double_as_longlong(cf), y = __double_as_longlong(bee[i]);
    return __longlong_as_double(x < y ? x : y);
}

// FP64 sweep of one ray with any number of emitting points (m0, m1) by a pair
// of lanes of one warp (gl = 0, 1; gmask = the pair).  ba holds the ray's raw
// alpha deposits, or after prepare_ray (`ready`; always with e) its loss
// coefficients, bee then the limits on the loss; be its raw eps deposits.
// Lane gl owns the ray's source points j with j %
// 2 == gl and keeps their photon rates Phi_j (FP64, in place of their eps
// slots); the total flux of a segment (zeta_s, zeta_d) is summed over the
// pair with one shuffle.  The loss of source j over segment i is R_ij =
// (alpha_i + alpha_{i+1}) G_ij zeta_d zeta_s with G_ij = (1/2) dV_ij
// zeta_g,ij (Eq. 14-16), and Phi_j <- max(Phi_j - R_ij, 0) (Eq. 13) is one
// FMA and a test of the sign bit.  Bound by the FP64 units: three
// instructions per source and segment.  Both lanes return F_0.
constexpr uint64_t EVEN_BITS = 0x5555555555555555ull;   // bits j with j % 2 == 0

template <int MODE>
__device__ __forceinline__ double sweep_ray(const WalkArgs& a, const double* ba, double* be, const double* bee,
                                            const Scales& sc, uint64_t m0, uint64_t m1, int gl, unsigned gmask, bool ready) {
    const int nr = a.nr;
    const uint64_t sel = EVEN_BITS << gl;                     // the lane's parity (64 is even)
    uint64_t o0 = m0 & sel, o1 = m1 & sel;                    // own live sources
    const double f4pi = (MODE == 0 ? 1.0 : 1.0 / (double)sc.eps) * (1.0 / (4.0 * PI_D));
    for (uint64_t w = o0; w; w &= w - 1) { const int j = __ffsll((long long)w) - 1; be[j] = bin_value<MODE>(be + j, f4pi); }
    for (uint64_t w = o1; w; w &= w - 1) { const int j = 64 + __ffsll((long long)w) - 1; be[j] = bin_value<MODE>(be + j, f4pi); }
    double* ph = be;                                              // Eq. 12
    const int jtop = farthest(m0, m1), ia = unit_base(sc.a);
    double a_hi = ready ? 0.0 : alpha_at<MODE>(a, ba, jtop, ia);
    for (int i = jtop - 1; i >= 0; --i) {
        double A = ba[i];
        if (!ready) {                                             // (in the shadow of the FP64 chain)
            const double a_lo = alpha_at<MODE>(a, ba, i, ia);
            A = a_lo + a_hi;
            a_hi = a_lo;
        }
        const int b = i + 1;                                      // sources strictly beyond r_i
        const uint64_t a0 = (b < 64) ? (o0 & (~0ull << b)) : 0ull;
        const uint64_t a1 = (b <= 64) ? o1 : (o1 & (~0ull << (b - 64)));
        const double* id2 = a.ID2 + (size_t)i * nr;
        const double* gi = a.GI + (size_t)i * nr;
        double Fl = 0.0;                                          // Eq. 11 at the segment midpoint
        for (uint64_t w = a0; w; w &= w - 1) { const int j = __ffsll((long long)w) - 1; Fl = fma(ph[j], __ldg(id2 + j), Fl); }
        for (uint64_t w = a1; w; w &= w - 1) { const int j = 64 + __ffsll((long long)w) - 1; Fl = fma(ph[j], __ldg(id2 + j), Fl); }
        const double Ftot = Fl + __shfl_xor_sync(gmask, Fl, 1);
        if (positive(Ftot)) {
            const double cf = loss_coef(A * recip(Ftot), bee, i);   // zeta_s = F_j / Ftot (Eq. 16)
            for (uint64_t w = a0; w; w &= w - 1) {
                const int j = __ffsll((long long)w) - 1;
                const double np = fma(-cf * __ldg(gi + j), ph[j], ph[j]);   // Eq. 13-14
                if (positive(np)) ph[j] = np; else { ph[j] = 0.0; o0 &= ~(1ull << j); }
            }
            for (uint64_t w = a1; w; w &= w - 1) {
                const int j = 64 + __ffsll((long long)w) - 1;
                const double np = fma(-cf * __ldg(gi + j), ph[j], ph[j]);
                if (positive(np)) ph[j] = np; else { ph[j] = 0.0; o1 &= ~(1ull << (j - 64)); }
            }
        } else if (!__any_sync(gmask, (o0 | o1) != 0ull)) {
            break;                                                // nothing left beyond or before r_i on the ray
        }
    }
    double F0 = 0.0;                                              // Eq. 10-11 at r = 0
    for (uint64_t w = o0; w; w &= w - 1) { const int j = __ffsll((long long)w) - 1; F0 = fma(ph[j], __ldg(a.inv_r2 + j), F0); }
    for (uint64_t w = o1; w; w &= w - 1) { const int j = 64 + __ffsll((long long)w) - 1; F0 = fma(ph[j], __ldg(a.inv_r2 + j), F0); }
    return F0 + __shfl_xor_sync(gmask, F0, 1);
}

// The sweep of the FP32 form.  The deposits (alpha, e) and the geometric
// factors are FP32 quantities, so each segment's loss R_ij (Eq. 14) is formed
// in FP32.  The emitted budget E_j = eps_j / 4pi (Eq. 12) and the running loss
// L_j = sum of R_ij are carried as unevaluated sums of two FP32 numbers
// (hi + lo, about 48 significant bits; L by compensated addition), so that
// the per-segment work needs no FP64 instruction -- on GB300 FP64 runs at
// 1/64 of the FP32 rate and would make the sweep cost grow with the number
// of sources on a ray.  A source is spent when L_j reaches E_j
// (Phi = max(E - L, 0), Eq. 13).  The cancellation Phi_j = E_j - L_j that
// decides the flux near the ionisation front, the flux F_0 (Eq. 10-11) and
// hence the ionised/neutral classification are done in FP64 at the end of
// the ray.
__device__ __forceinline__ float2 two_sum(float a, float b) {    // Knuth: a + b = s + e exactly
    const float s = a + b;
    const float bp = s - a;
    const float e = (a - (s - bp)) + (b - bp);
    return make_float2(s, e);
}

__device__ __forceinline__ float phi_f(const float2 E, const float2 Lr) {  // E - L to FP32 precision
    return (E.x - Lr.x) + (E.y - Lr.y);
}

// FP32-form sweep of one ray by a group of SG lanes of one warp (gmask):
// lane gl owns the ray's source points j with j % SG == gl and keeps their
// budgets and losses; the total flux of each segment (for zeta_s, zeta_d) is
// summed over the group with shuffles.  All lanes of the group return F_0.
constexpr int SG = 2;
constexpr uint64_t SG_PATTERN = 0x5555555555555555ull;   // bits j with j % 2 == 0

__device__ __forceinline__ double sweep_ray_group(const WalkArgs& a, const double* ba, double* be, const double* bee,
                                  const Scales& sc, uint64_t m0, uint64_t m1, int gl, unsigned gmask) {
    const int nr = a.nr;
    if (!(m0 | m1)) return 0.0;
    const uint64_t sel = SG_PATTERN << gl;                    // 64 % SG == 0: same pattern for m1
    const uint64_t o0 = m0 & sel, o1 = m1 & sel;
    const double inv_eps = 1.0 / (double)sc.eps, inv4pi = 1.0 / (4.0 * PI_D);
    float2* E = reinterpret_cast<float2*>(be);
    float2* Ls = reinterpret_cast<float2*>(const_cast<double*>(ba));
    for (int half = 0; half < 2; ++half)
        for (uint64_t w = half ? o1 : o0; w; w &= w - 1) {
            const int j = (half ? 64 : 0) + __ffsll((long long)w) - 1;
            const double v = bin_value<1>(be + j, inv_eps) * inv4pi;   // Eq. 12
            const float hi = (float)v;
            E[j] = make_float2(hi, (float)(v - (double)hi));
        }
    const float ia = 1.0f / sc.a, ie = 1.0f / sc.e;
    const int jtop = m1 ? 64 + 63 - __clzll((long long)m1) : 63 - __clzll((long long)m0);
    float a_hi = bin_value_f<1>(ba + jtop, ia) * __ldg(a.inv_volf + jtop);
    __syncwarp(gmask);                                        // alpha at jtop read before any overwrite
    uint64_t d0 = 0, d1 = 0;                                  // own spent sources
    for (int i = jtop - 1; i >= 0; --i) {
        if (!__any_sync(gmask, ((o0 & ~d0) | (o1 & ~d1)) != 0ull)) break;
        const float a_lo = bin_value_f<1>(ba + i, ia) * __ldg(a.inv_volf + i);
        __syncwarp(gmask);                                    // everyone has read alpha_i
        const int b = i + 1;                                  // source b starts: its loss slot was alpha_b
        if (((b < 64 ? (o0 >> b) : (o1 >> (b - 64))) & 1ull)) Ls[b] = make_float2(0.f, 0.f);
        const uint64_t a0 = (b < 64) ? (o0 & ~d0 & (~0ull << b)) : 0ull;
        const uint64_t a1 = (b <= 64) ? (o1 & ~d1) : (o1 & ~d1 & (~0ull << (b - 64)));
        const float* id2 = a.ID2f + (size_t)i * nr;
        float Fl = 0.f;
        for (int half = 0; half < 2; ++half)
            for (uint64_t w = half ? a1 : a0; w; w &= w - 1) {
                const int j = (half ? 64 : 0) + __ffsll((long long)w) - 1;
                Fl = fmaf(phi_f(E[j], Ls[j]), __ldg(id2 + j), Fl);
            }
        int cnt = __popcll((long long)a0) + __popcll((long long)a1);
        for (int o = 1; o < SG; o <<= 1) {
            Fl += __shfl_xor_sync(gmask, Fl, o);
            cnt += __shfl_xor_sync(gmask, cnt, o);
        }
        if (cnt > 0) {
            const float A = a_lo + a_hi;                      // G carries the 1/2 of the mean
            const bool single = !bee && cnt == 1;             // zeta_s = 1, zeta_d = 1
            float cf = 0.f;
            bool go = true;
            if (!single) {
                if (Fl > 0.f) {
                    float zd = 1.f;                           // Eq. 17
                    if (bee) {
                        const float ev = bin_value_f<1>(bee + i + 1, ie) * __ldg(a.inv_volf + i + 1);
                        if (ev > 0.f) zd = fminf(2.f, __fdividef(Fl, ev));
                    }
                    cf = __fdividef(A * zd, Fl);              // zeta_s = F_j / Ftot (Eq. 16)
                } else {
                    go = false;
                }
            }
            if (go) {
                const float* gi = a.GIf + (size_t)i * nr;
                const float* g = a.Gf + (size_t)i * nr;
                for (int half = 0; half < 2; ++half)
                    for (uint64_t w = half ? a1 : a0; w; w &= w - 1) {
                        const int j = (half ? 64 : 0) + __ffsll((long long)w) - 1;
                        const float2 e = E[j];
                        const float2 L = Ls[j];
                        const float R = single ? A * __ldg(g + j) : cf * (__ldg(gi + j) * phi_f(e, L));   // Eq. 14
                        const float2 t = two_sum(L.x, R);     // compensated L += R
                        const float2 Ln = two_sum(t.x, t.y + L.y);
                        if (phi_f(e, Ln) > 0.f) Ls[j] = Ln;
                        else if (half) d1 |= 1ull << (j - 64); else d0 |= 1ull << j;   // spent: Phi = 0
                    }
            }
        }
        a_hi = a_lo;
    }
    double F0 = 0.0;                                          // Eq. 10-11 at r = 0, in FP64
    for (int half = 0; half < 2; ++half)
        for (uint64_t w = half ? (o1 & ~d1) : (o0 & ~d0); w; w &= w - 1) {
            const int j = (half ? 64 : 0) + __ffsll((long long)w) - 1;
            const float2 e = E[j];
            const float2 L = Ls[j];
            const double phi = ((double)e.x + (double)e.y) - ((double)L.x + (double)L.y);
            if (phi > 0.0) F0 = fma(phi, __ldg(a.inv_r2 + j), F0);
        }
    for (int o = 1; o < SG; o <<= 1) F0 += __shfl_xor_sync(gmask, F0, o);
    return F0;
}

// Per-target ray tables for the sweep, in shared scratch: cls (per chunk of 16
// rays and class, the rays of that class, one bit per two lanes), npts (per
// chunk, emitting points), order (u16, the ray of each rank), off (u16, first
// lane of each lane group), m1 (emitting points 64 and beyond, with N_R > 64
// only).
constexpr int MAX_NPIX = 12 * 8 * 8;                  // N_side <= 8
constexpr int GROUP_MAX = 32;                         // rays with more points go to lane pairs
constexpr int GROUP_MEAN_MAX = 14;                    // lane groups while a lit ray has at most this many points on average
// FP64 sweeps: lane groups while a target's fill at most this many lanes (see
// sweep_rays)
__device__ __forceinline__ int group_lanes_max(int npix) { return max(128, 4 * npix / 3); }
constexpr int N_CLS = 7;                              // classes of rays with emitting points
struct RayScratch {
    uint32_t* cls;
    int* npts;
    uint64_t* m1;
    uint16_t *order, *off;
};
__host__ __device__ constexpr size_t ray_chunks(int npix) { return ((size_t)npix + 15) / 16; }
__host__ __device__ constexpr size_t sweep_scratch_bytes(int npix, int nr) {
    return (nr > 64 ? (size_t)npix * 8 : 0) + ray_chunks(npix) * (N_CLS + 1) * 4 + (size_t)npix * 4;
}
__device__ __forceinline__ RayScratch ray_scratch(unsigned char* p, int npix, int nr) {
    RayScratch rs;
    rs.m1 = reinterpret_cast<uint64_t*>(p);
    rs.cls = reinterpret_cast<uint32_t*>(p + (nr > 64 ? (size_t)npix * 8 : 0));
    rs.npts = reinterpret_cast<int*>(rs.cls + ray_chunks(npix) * N_CLS);
    rs.order = reinterpret_cast<uint16_t*>(rs.npts + ray_chunks(npix));
    rs.off = rs.order + npix;
    return rs;
}

// The emitting points of ray k, as ray_census left them: points below 64 in
// the ray's eps slot 0 (a deposit there is at the target itself and not swept).
__device__ __forceinline__ void ray_mask(const double* bins_eps, const RayScratch& rs, int nr, int k, uint64_t& m0,
                                         uint64_t& m1) {
    m0 = *reinterpret_cast<const uint64_t*>(bins_eps + (size_t)k * nr);
    m1 = nr > 64 ? rs.m1[k] : 0ull;
}

// Lanes given to a ray with c emitting points in a lane group: the next
// power of two.
__device__ __forceinline__ int group_width(int c) { return c <= 1 ? c : 1 << (32 - __clz(c - 1)); }

// Class of a ray by its emitting points c: 0 more than GROUP_MAX, then by
// decreasing group width 32, 16, .. 1; -1: no points.
__device__ __forceinline__ int ray_class(int c) {
    if (c == 0) return -1;
    return c > GROUP_MAX ? 0 : 1 + __clz(c == 1 ? 1 : 2 * c - 1) - 26;
}

struct Ranks { int nz, lanes, nbig, none, npts; };    // rays with points, lanes of the groups, rays of more than
                                                      // GROUP_MAX points and of one point, points of all rays

// Finds each ray's emitting points (a lane pair per ray) and ranks the rays
// by class, ties by ray index: deterministic, so that sums over the rays are.
// The lane groups, sorted by decreasing power-of-two width, never straddle a
// warp.  Two barriers, no loop over the other rays
// (counting by one thread per ray and comparing all pairs of rays took 3 k
// warp instructions per target at N_PIX 48).
template <int MODE, int NT>
__device__ __forceinline__ Ranks rank_rays(const WalkArgs& a, double* bins_eps, const RayScratch& rs) {
    const int npix = a.npix, nr = a.nr, tid = threadIdx.x, lane = tid & 31, gl = tid & 1;
    for (int k = tid >> 1; k < (int)ray_chunks(npix) * 16; k += NT / 2) {   // warp-uniform: 16 rays
        uint64_t m0 = 0, m1 = 0;
        double* be = bins_eps + (size_t)k * nr;
        if (k < npix)
            for (int j = 2 - gl; j < nr; j += 2)               // lane gl scans its parity (j >= 1)
                if (bin_nonzero<MODE>(be + j)) { if (j < 64) m0 |= 1ull << j; else m1 |= 1ull << (j - 64); }
        m0 |= __shfl_xor_sync(FULL, m0, 1);
        m1 |= __shfl_xor_sync(FULL, m1, 1);
        const int c = __popcll((long long)m0) + __popcll((long long)m1);
        const int cls = ray_class(c), chunk = k >> 4;
        const int sum = __reduce_add_sync(FULL, gl ? 0 : c);
        if (k < npix && gl == 0) {
            *reinterpret_cast<uint64_t*>(be) = m0;
            if (nr > 64) rs.m1[k] = m1;
        }
        for (int q = 0; q < N_CLS; ++q) {
            const unsigned m = __ballot_sync(FULL, cls == q && gl == 0);
            if (lane == 0) rs.cls[chunk * N_CLS + q] = m;
        }
        if (lane == 0) rs.npts[chunk] = sum;
    }
    __syncthreads();                                          // masks and class bits visible
    const int nch = (int)ray_chunks(npix);
    Ranks r{0, 0, 0, 0, 0};
    for (int ch = 0; ch < nch; ++ch) {
        r.npts += rs.npts[ch];
        for (int q = 0; q < N_CLS; ++q) {
            const int n = __popc(rs.cls[ch * N_CLS + q]);
            r.nz += n;
            if (q == 0) r.nbig += n;
            else r.lanes += n << (6 - q);
            if (q == N_CLS - 1) r.none += n;
        }
    }
    for (int k = tid; k < npix; k += NT) {
        uint64_t m0, m1;
        ray_mask(bins_eps, rs, nr, k, m0, m1);
        const int cls = ray_class(__popcll((long long)m0) + __popcll((long long)m1));
        if (cls < 0) continue;
        int rank = 0, lanes = 0;
        for (int ch = 0; ch < nch; ++ch)
            for (int q = 0; q <= cls; ++q) {
                unsigned m = rs.cls[ch * N_CLS + q];
                if (q == cls && ch >= (k >> 4)) m = ch > (k >> 4) ? 0u : m & ((1u << (2 * (k & 15))) - 1u);
                const int n = __popc(m);
                rank += n;
                if (q > 0) lanes += n << (6 - q);
            }
        rs.order[rank] = (uint16_t)k;
        rs.off[rank] = (uint16_t)lanes;
    }
    __syncthreads();                                          // ranks visible
    return r;
}

// The lane group that group-lane p of T belongs to: its ray k, the ray's points
// c, the group's width w, the lane's place in it, its own point jA (0: none)
// and the ray's farthest.  Returns whether p < T.
__device__ __forceinline__ bool group_lane(const double* bins_eps, const RayScratch& rs, const Ranks& rk, int nr, int p, int T,
                                           int& k, int& c, int& w, int& slot, int& jA, int& jtop) {
    const bool in = p < T;
    int g = rk.nbig;                                          // the last rank whose group starts at or before p
    uint64_t m0 = 0, m1 = 0;
    k = slot = 0;
    if (in) {
        int hi = rk.nz - 1;
        while (g < hi) {
            const int mid = (g + hi + 1) >> 1;
            if ((int)rs.off[mid] <= p) g = mid; else hi = mid - 1;
        }
        k = rs.order[g];
        slot = p - (int)rs.off[g];
        ray_mask(bins_eps, rs, nr, k, m0, m1);
    }
    c = __popcll((long long)m0) + __popcll((long long)m1);
    w = group_width(c);
    jtop = farthest(m0, m1);
    for (int n = 0; n < slot; ++n) { if (m0) m0 &= m0 - 1; else m1 &= m1 - 1; }
    jA = m0 ? __ffsll((long long)m0) - 1 : (m1 ? 63 + __ffsll((long long)m1) : 0);
    return in;
}

// FP64 sweep, after prepare_ray, of 32 group lanes from `base` on: a lane per
// emitting point of the rays with up to GROUP_MAX points, its Phi_j in a
// register, the segments far to near in lockstep over the warp.  A segment's
// total flux is a butterfly sum over the group.  The tables hold zero for
// points not beyond the segment and a spent source is zero, so nothing is
// masked.  6 + log2(w) FP64 instructions per segment for 32 points; the tables
// are loaded a segment ahead.  Each group's first lane returns its ray's F_0.
template <int MODE>
__device__ __forceinline__ double sweep_group64(const WalkArgs& a, const double* bins_a, const double* bins_eps,
                                                const double* bins_e, const Scales& sc, const RayScratch& rs,
                                                const Ranks& rk, int base, int T) {
    const int nr = a.nr, lane = threadIdx.x & 31;
    int k, c, w, slot, jA, jtop;
    const bool in = group_lane(bins_eps, rs, rk, nr, base + lane, T, k, c, w, slot, jA, jtop);
    const double* ba = bins_a + (size_t)k * nr;
    const double* bee = bins_e ? bins_e + (size_t)k * nr : nullptr;
    double ph = 0.0;
    if (jA > 0) ph = bin_value<MODE>(bins_eps + (size_t)k * nr + jA, (MODE == 0 ? 1.0 : 1.0 / (double)sc.eps) * (1.0 / (4.0 * PI_D)));
    const int wmax = __reduce_max_sync(FULL, (unsigned)w);
    const int itop = __reduce_max_sync(FULL, (unsigned)jtop);
    const double* id2p = a.ID2 + (size_t)(itop - 1) * nr + jA;
    const double* gip = a.GI + (size_t)(itop - 1) * nr + jA;
    double id2 = __ldg(id2p), gi = __ldg(gip);
    for (int i = itop - 1; i >= 0; --i) {
        const double id2c = id2, gic = gi;
        if (i > 0) { id2p -= nr; gip -= nr; id2 = __ldg(id2p); gi = __ldg(gip); }
        double F = ph * id2c;                                 // Eq. 11 at the segment midpoint
        for (int o = 1; o < wmax; o <<= 1) {
            const double t = __shfl_xor_sync(FULL, F, o);
            if (o < w) F += t;
        }
        if (positive(F)) {
            const double cf = loss_coef(ba[i] * recip(F), bee, i);   // zeta_s = F_j / F_tot (Eq. 16)
            const double np = fma(-cf * gic, ph, ph);         // Eq. 13-14
            ph = positive(np) ? np : 0.0;
        }
        if (!__any_sync(FULL, positive(ph))) break;           // every point of the warp spent
    }
    double F0 = ph * __ldg(a.inv_r2 + jA);                    // Eq. 10-11 at r = 0
    for (int o = 1; o < wmax; o <<= 1) {
        const double t = __shfl_xor_sync(FULL, F0, o);
        if (o < w) F0 += t;
    }
    return in && slot == 0 ? F0 : 0.0;
}

// Double-FP32 sweep of the rays of a target with 1..GROUP_MAX emitting
// points, a lane per point (a lane per point spends less on bookkeeping than
// a lane pair looping over a ray's points, but idles on the points not yet
// reached; it wins while rays carry few points): the rays' lane groups (rank order, group_width
// lanes each) are laid end to end over the CTA's warps, and lane `slot` of a
// ray's group keeps the ray's slot-th emitting point in registers: its
// budget E_j = eps_j / 4pi and running loss L_j as unevaluated FP32 pairs
// (Eq. 12-14, as in sweep_ray_group), with the segments swept far to near in
// lockstep over the warp.  A segment's total flux (zeta_s, zeta_d; Eq.
// 16-17) is a butterfly sum over the group, the same in every lane of it.  A
// ray with one point and no e has zeta_s = zeta_d = 1, R_ij = A_i G_ij.
// Each group's first lane returns its ray's F_0 (FP64) in the sum.
template <int NT>
__device__ __forceinline__ double sweep_groups(const WalkArgs& a, const double* bins_a, const double* bins_eps, const double* bins_e,
                               const Scales& sc, const RayScratch& rs, const Ranks& rk) {
    const int nr = a.nr, lane = threadIdx.x & 31, T = rk.lanes;
    const double inv_eps = 1.0 / (double)sc.eps, inv4pi = 1.0 / (4.0 * PI_D);
    const float ia = 1.0f / sc.a, ie = 1.0f / sc.e;
    double Fk = 0.0;
    for (int base = threadIdx.x & ~31; base < T; base += NT) {  // warp-uniform
        int k, c, w, slot, jA, jtop;
        const bool in = group_lane(bins_eps, rs, rk, nr, base + lane, T, k, c, w, slot, jA, jtop);
        const double* ba = bins_a + (size_t)k * nr;
        const double* be = bins_eps + (size_t)k * nr;
        const double* bee = bins_e ? bins_e + (size_t)k * nr : nullptr;
        const bool vA = slot < c;
        float2 EA = make_float2(0.f, 0.f), LA = EA;
        if (vA) { const double v = bin_value<1>(be + jA, inv_eps) * inv4pi; EA.x = (float)v; EA.y = (float)(v - (double)EA.x); }
        bool sA = !vA;                                        // spent, or no point
        const bool single = c == 1 && !bee;                   // zeta_s = zeta_d = 1 throughout
        const int wmax = __reduce_max_sync(FULL, (unsigned)w);
        const int itop = __reduce_max_sync(FULL, (unsigned)jtop);
        auto alpha = [&](int i) { return in ? bin_value_f<1>(ba + i, ia) * __ldg(a.inv_volf + i) : 0.f; };
        // the tables and the coefficient of a segment are fetched one segment
        // ahead of the chain F_tot -> R -> Phi
        const float* id2p = a.ID2f + (size_t)(itop - 1) * nr + jA;
        const float* gp = (single ? a.Gf : a.GIf) + (size_t)(itop - 1) * nr + jA;
        float a_hi = alpha(itop), a_nx = alpha(itop - 1), id2n = __ldg(id2p), gn = __ldg(gp);
        for (int i = itop - 1; i >= 0; --i) {
            if (!__any_sync(FULL, !sA)) break;                // every point of the warp spent
            const float a_lo = a_nx, id2 = id2n, g = gn;
            if (i > 0) { id2p -= nr; gp -= nr; id2n = __ldg(id2p); gn = __ldg(gp); a_nx = alpha(i - 1); }
            const bool live = !sA && jA > i;
            const float ph = live ? phi_f(EA, LA) : 0.f;
            float Fl = live ? ph * id2 : 0.f;                 // Eq. 11 at the segment midpoint
            for (int o = 1; o < wmax; o <<= 1) {
                const float t = __shfl_xor_sync(FULL, Fl, o);
                if (o < w) Fl += t;
            }
            if (live) {                                       // then Fl > 0
                const float A = a_lo + a_hi;                  // G carries the 1/2 of the mean
                float R;
                if (single) {
                    R = A * g;                                // Eq. 14
                } else {
                    float zd = 1.f;                           // Eq. 17
                    if (bee) {
                        const float ev = bin_value_f<1>(bee + i + 1, ie) * __ldg(a.inv_volf + i + 1);
                        if (ev > 0.f) zd = fminf(2.f, __fdividef(Fl, ev));
                    }
                    R = __fdividef(A * zd, Fl) * (g * ph);    // zeta_s = F_j / Ftot
                }
                const float2 t = two_sum(LA.x, R);            // compensated L += R
                const float2 Ln = two_sum(t.x, t.y + LA.y);
                if (phi_f(EA, Ln) > 0.f) LA = Ln; else sA = true;   // spent: Phi = 0 (Eq. 13)
            }
            a_hi = a_lo;
        }
        double F0 = 0.0;                                      // Eq. 10-11 at r = 0, in FP64
        if (!sA) {
            const double phi = ((double)EA.x + (double)EA.y) - ((double)LA.x + (double)LA.y);
            if (phi > 0.0) F0 = fma(phi, __ldg(a.inv_r2 + jA), F0);
        }
        for (int o = 1; o < wmax; o <<= 1) {
            const double t = __shfl_xor_sync(FULL, F0, o);
            if (o < w) F0 += t;
        }
        if (in && slot == 0) Fk += F0;
    }
    return Fk;
}

// Sum over the rays of one target (Eq. 18), ranked by rank_rays; `turn`
// rotates which warps take the work from target to target.
// FP64 sweeps (FP64 form and FP32 + FP64-sweep form): rays with a lone source
// by a warp each (lone_ray).  Of the others, while their points fill at most
// group_lanes_max lanes, all warps ready the rays (prepare_ray) and sweep them a
// lane per point (sweep_group64; more than GROUP_MAX points: lane pairs): the
// fewest FP64 instructions in a row, and the target's time is that chain.  Beyond that the FP64 units are what is short,
// and lane pairs, 16 rays of like load to a warp, take fewest in all (a lane
// for a point that the sweep has not reached costs as much as a busy one).
// The line lies at 128 lanes for up to 96 rays (turbulent128 278 -> 236 ms
// with it, 275 with pairs only, 251 with 64 lanes) and at 4/3 of a lane per ray
// beyond (N_PIX 192, 64^3, 10 sources: 23.1 ms with 256 lanes, 23.9 with 128;
// AMR 64^3 24 ms, 35 with groups only).  Coefficients computed within the chain
// where lane pairs sweep: 505 -> 492 ms for 10^4 sources at 128^3 (its FP64
// units are busy).
// Double-FP32 sweep: lane groups up to GROUP_MEAN_MAX points per lit ray on
// average (sweep_groups), lane pairs beyond (sweep_ray_group).  The choices
// depend only on the bins and N_PIX, so a target's rays are swept alike in a CTA
// of any size, alone, in a batch or from stored bins; only the order of the sum
// over the rays follows the CTA.  `scratch` holds sweep_scratch_bytes bytes of
// shared memory; all threads call.
template <int MODE, int NT>
__device__ __forceinline__ double sweep_rays(const WalkArgs& a, double* bins_a, double* bins_eps, double* bins_e,
                                             const Scales& sc, unsigned char* scratch, int turn) {
    const int nr = a.nr, tid = threadIdx.x, lane = tid & 31;
    constexpr int NW = NT / 32;
    const RayScratch rs = ray_scratch(scratch, a.npix, nr);
    const bool use_e = a.use_e != 0;
    const Ranks rk = rank_rays<MODE, NT>(a, bins_eps, rs);
    double Fk = 0.0;
    uint64_t m0 = 0, m1 = 0;
    if constexpr (MODE != 2) {
        const int wid = ((tid >> 5) + turn) & (NW - 1);       // its place in the sum too (block_sum)
        const int n_lone = use_e ? 0 : rk.none, T = rk.lanes - n_lone, n_more = rk.nz - n_lone;
        const bool groups = T <= group_lanes_max(a.npix), ready = groups || use_e;
        for (int r = (ready ? 0 : n_more) + wid; r < rk.nz; r += NW) {
            const int k = rs.order[r];
            ray_mask(bins_eps, rs, nr, k, m0, m1);
            const int jtop = farthest(m0, m1);
            if (r < n_more) prepare_ray<MODE>(a, bins_a + k * nr, use_e ? bins_e + k * nr : nullptr, sc, jtop);
            else Fk += lone_ray<MODE>(a, bins_a + k * nr, bins_eps + k * nr, sc, jtop);
        }
        if (ready) __syncthreads();                           // coefficients visible
        const int n_pair = groups ? rk.nbig : n_more;
        const int gl = tid & 1;
        const unsigned gmask = 3u << (lane & ~1);
        for (int r = wid * 16 + (lane >> 1); r < n_pair; r += NT / 2) {
            const int k = rs.order[r];
            ray_mask(bins_eps, rs, nr, k, m0, m1);
            const double f = sweep_ray<MODE>(a, bins_a + k * nr, bins_eps + k * nr, use_e ? bins_e + k * nr : nullptr,
                                             sc, m0, m1, gl, gmask, ready);
            if (gl == 0) Fk += f;
        }
        if (groups)
            for (int base = (NW - 1 - wid) * 32; base < T; base += NT)
                Fk += sweep_group64<MODE>(a, bins_a, bins_eps, use_e ? bins_e : nullptr, sc, rs, rk, base, T);
        return Fk;
    } else {
    const int gl = tid % SG;
    const unsigned gmask = ((1u << SG) - 1u) << (lane & ~(SG - 1));
    if (rk.npts > GROUP_MEAN_MAX * rk.nz) {
        // many points per ray: every ray by lane pairs, in ray order (ranked
        // order would put the heaviest rays in one warp, which then holds
        // the CTA's barrier)
        for (int k = tid / SG; k < a.npix; k += NT / SG) {
            ray_mask(bins_eps, rs, nr, k, m0, m1);
            const double f = sweep_ray_group(a, bins_a + k * nr, bins_eps + k * nr, use_e ? bins_e + k * nr : nullptr,
                                             sc, m0, m1, gl, gmask);
            if (gl == 0) Fk += f;
        }
        return Fk;
    }
    // the pair-swept rays round-robin over the warps, so that no warp holds
    // the CTA's barrier with all of them
    for (int r = (tid >> 5) + NW * (lane / SG); r < rk.nbig; r += NT / SG) {
        const int k = rs.order[r];
        ray_mask(bins_eps, rs, nr, k, m0, m1);
        const double f = sweep_ray_group(a, bins_a + k * nr, bins_eps + k * nr, use_e ? bins_e + k * nr : nullptr,
                                         sc, m0, m1, gl, gmask);
        if (gl == 0) Fk += f;
    }
    return Fk + sweep_groups<NT>(a, bins_a, bins_eps, use_e ? bins_e : nullptr, sc, rs, rk);
    }
}

template <int NT>
__device__ __forceinline__ double block_sum(double v, double* red, int turn) {
    v = warp_sum(v);                                               // (the sum's order follows the rotated warps)
    const int lane = threadIdx.x & 31, wid = ((threadIdx.x >> 5) + turn) & (NT / 32 - 1);
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < NT / 32; ++w) t += red[w];
    return t;                                                      // valid in thread 0
}

// Per-thread walk counters go to the job's counters (one atomic per warp).  A
// thread counts at most some 3e7 table entries for one target (512^3, every cell
// and its seven mirror images accepted), so 32 bits hold those of 64.
constexpr unsigned FLUSH_TARGETS = 64;
struct WalkCounters {
    unsigned vis = 0, acc = 0, ent = 0;     // (flushed every FLUSH_TARGETS targets, before they can wrap)
    unsigned fb_mac = 0, fb_dep = 0;        // FP32 forms: decisions re-taken in FP64
};

__device__ __forceinline__ void flush_counters(const WalkArgs& a, WalkCounters& c) {
    unsigned long long fm = c.fb_mac, fd = c.fb_dep, vis = c.vis, acc = c.acc, ent = c.ent;
    for (int o = 16; o > 0; o >>= 1) {
        vis += __shfl_xor_sync(FULL, vis, o);
        acc += __shfl_xor_sync(FULL, acc, o);
        ent += __shfl_xor_sync(FULL, ent, o);
        fm += __shfl_xor_sync(FULL, fm, o);
        fd += __shfl_xor_sync(FULL, fd, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(a.stats + 0, vis);
        atomicAdd(a.stats + 1, acc);
        atomicAdd(a.stats + 2, ent);
        if (fm) atomicAdd(a.stats + 3, fm);
        if (fd) atomicAdd(a.stats + 4, fd);
    }
    c = WalkCounters();
}

// One CTA of NT threads per target, persistent over the targets of a list of
// jobs (a job = one tree and a range or list of its cells).  Several trees in
// one launch is how independent requests are batched together.  Each step
// pops NT/8 opened nodes and evaluates their NT children, one per thread.
// VAR: the kernel choices other than W_p / W_f,3 and the periodic and
// corner-of-symmetry boundaries are compiled in (a separate instantiation,
// so that the default walk keeps its registers).
// OUT: OUT_FUSED walk + map + sweep; OUT_DUMP keeps the raw bins and
// accepted ids; OUT_CD column-density maps (no radial points, no sweep).
constexpr int OUT_FUSED = 0, OUT_DUMP = 1, OUT_CD = 2;

// A target cell: its corner and edge (finest cells) and centre.
template <int MODE>
struct Target {
    typename Prec<MODE>::real px, py, pz;
    int tx, ty, tz, ts;
};

// Where a node lies as seen from the target, in the copy that the boundary
// puts there: offset o = 2 (node centre - target centre) in half cells, and
// the squared distance of its centre of mass (FP32 forms: within B of the
// FP64 value).
template <int MODE>
struct NodeView {
    typename Prec<MODE>::real qx, qy, qz, d2;
    float B;
    int ox, oy, oz;
};

template <int MODE, bool VAR>
__device__ __forceinline__ NodeView<MODE> view_node(const WalkArgs& a, const Target<MODE>& t, int img, int cx, int cy,
                                                    int cz, int s, const typename Prec<MODE>::real* cm, float kap) {
    using real = typename Prec<MODE>::real;
    NodeView<MODE> v;
    v.ox = 2 * cx + s - 2 * t.tx - t.ts; v.oy = 2 * cy + s - 2 * t.ty - t.ts; v.oz = 2 * cz + s - 2 * t.tz - t.ts;
    v.qx = t.px; v.qy = t.py; v.qz = t.pz;
    if (VAR && a.bc != TR_BC_ISOLATED) {
        bc_frame<real>(a.bc, img & 1, a.N, 2 * cx + s, 2 * t.tx + t.ts, t.px, v.ox, v.qx);
        bc_frame<real>(a.bc, (img >> 1) & 1, a.N, 2 * cy + s, 2 * t.ty + t.ts, t.py, v.oy, v.qy);
        bc_frame<real>(a.bc, (img >> 2) & 1, a.N, 2 * cz + s, 2 * t.tz + t.ts, t.pz, v.oz, v.qz);
    }
    if constexpr (MODE == 0) {
        v.d2 = dist2(v.qx, v.qy, v.qz, cm);
        v.B = 0.f;
    } else {
        // centre of mass - target = o/2 + offset (a mirror image of the corner
        // of symmetry mirrors the offset too)
        const bool mir = VAR && a.bc == TR_BC_CORNER;
        const float ex = fmaf(0.5f, (float)v.ox, (mir && (img & 1)) ? -cm[0] : cm[0]);
        const float ey = fmaf(0.5f, (float)v.oy, (mir && (img & 2)) ? -cm[1] : cm[1]);
        const float ez = fmaf(0.5f, (float)v.oz, (mir && (img & 4)) ? -cm[2] : cm[2]);
        v.d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
        v.B = d2_err_bound(v.d2, kap * (float)s);
    }
    return v;
}

struct Bins {
    double *a, *eps, *e;                    // e: only with e_prev
};

// Map and spread up to 32 accepted nodes onto the target's rays, by one warp
// and without a barrier of the CTA.  First a lane per node: its table key,
// its ray entries and its radial weights.  Then a lane per (node, ray) pair,
// the pairs of all 32 nodes laid end to end: a lane finds its node from the
// bit mask of the pairs that start a node, loads the table entry a round
// ahead, and adds to the node's points on that ray.  Both halves keep the
// lanes full, which a thread that evaluates a node and then spreads it
// cannot: at theta = 0.5 three quarters of the evaluated nodes are accepted,
// and a node has 1 to 20 rays and 1 to 10 points.
template <int MODE, int OUT, bool VAR, int W>
__device__ __forceinline__ void spread_nodes(const WalkArgs& a, NodeBatch<MODE, W>& nb, uint32_t entry, bool have, int img,
                                             const Target<MODE>& t, const Bins& bins, const Scales& sc, float kap,
                                             WalkCounters& cnt) {
    using real = typename Prec<MODE>::real;
    constexpr bool CD = OUT == OUT_CD;
    const int lane = threadIdx.x & 31, nr = a.nr;
    const bool use_e = a.use_e != 0;
    const uint32_t* const tent = a.tent;
    int ne = 0, eps_i = 0;
    uint32_t off = 0;
    RadialSpread<MODE> n;
    n.b = real(1); n.lo = 0; n.npts = 0; n.lng = false;
    real alpha = real(0), e = real(0), eps = real(0), w1 = real(0);
    double md = 0.0;
    if (have) {
        const int lev = (int)(entry >> 27);
        const uint32_t mort = entry & 0x7ffffffu;
        const int s = a.N >> lev;
        const int cx = (int)compact3(mort) * s, cy = (int)compact3(mort >> 1) * s, cz = (int)compact3(mort >> 2) * s;
        const int64_t nid = level_offset(lev) + mort;
        real cm[3], m, qv[3], mion;
        load_node<MODE>(a.nodes, nid, cm, m, qv, mion);
        const NodeView<MODE> v = view_node<MODE, VAR>(a, t, img, cx, cy, cz, s, cm, kap);
        const real d = sqrt(v.d2);
        if (CD) {
            const uint2 hd = __ldg(a.hdr + table_key(v.ox, v.oy, v.oz, s));
            off = hd.x; ne = (int)hd.y;
            md = (double)m / (a.cd_omega * ((double)d * (double)d));
            cnt.ent += ne;
        } else {
            // FP32 forms: |d - d64| <= dtol; the choices that jump with d and
            // lie closer than that are taken on d64
            const float dtol = MODE != 0 ? __fdividef(v.B, (float)d) + 4.f * U32 * (float)d : 0.f;
            double d64 = -1.0;
            auto exact_d = [&]() -> double {
                if (d64 < 0.0) { d64 = sqrt(exact_d2(a, nid, v.qx, v.qy, v.qz)); ++cnt.fb_dep; }
                return d64;
            };
            bool in_reach;
            if constexpr (MODE == 0) {
                in_reach = !less(a.lray, d);
            } else {
                if ((float)d + dtol < a.lrayf * (1.f - 2.f * U32)) in_reach = true;
                else if ((float)d - dtol > a.lrayf * (1.f + 2.f * U32)) in_reach = false;
                else in_reach = exact_d() <= a.lray;
            }
            if (in_reach) {
                const uint2 hd = __ldg(a.hdr + table_key(v.ox, v.oy, v.oz, s));
                off = hd.x; ne = (int)hd.y;
                cnt.ent += ne;
                if (MODE == 0 ? positive(qv[1]) : qv[1] != real(0)) {
                    if (VAR && a.kern_e != TR_EPS_WF3) {
                        const double dvar = MODE != 0 ? exact_d() : (double)d;
                        deposit_eps_variant<MODE>(a, bins.eps, off, ne, dvar, qv[1], sc.eps, s);
                    } else {
                        eps = qv[1];
                        eps_i = eps_split<MODE>(a, d, w1);
                    }
                }
                if (qv[0] != real(0) || (a.use_e && qv[2] != real(0))) {
                    const int gauss = VAR ? a.kern_a : 0;
                    real* const wcol = &nb.w[0][lane];
                    if constexpr (MODE == 0) radial_setup64<W>(a, n, d, s, wcol, gauss);
                    else if (radial_setup<MODE, W>(a, n, d, s, wcol, gauss, dtol))
                        radial_setup_exact<MODE>(a, n, exact_d(), s, wcol, gauss);
                    alpha = qv[0];
                    e = a.use_e ? qv[2] : real(0);
                    if constexpr (MODE != 0) {               // a fixed-point bin takes no addend below +0 (nor -0, NaN)
                        alpha = alpha > 0.f ? alpha : 0.f;
                        e = e > 0.f ? e : 0.f;
                    }
                }
            }
        }
    }
    // the batch's (node, ray) pairs, end to end
    const bool act = ne > 0 && (CD || n.npts > 0 || eps != real(0));
    if (!act) ne = 0;
    int incl = ne;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(FULL, incl, 31), start = incl - ne;
    const unsigned am = __ballot_sync(FULL, act), lt = (1u << lane) - 1u;
    if (act) {
        const int k = __popc(am & lt);
        nb.key[k] = make_uint2(off - (uint32_t)start,
                               (uint32_t)n.lo | ((uint32_t)n.npts << 7) | ((uint32_t)lane << 15) |
                                   ((uint32_t)eps_i << 20) | (eps != real(0) ? PK_EPS : 0u) | (n.lng ? PK_LONG : 0u));
        if constexpr (CD) {
            reinterpret_cast<double*>(&nb.w[0][0])[k] = md;
        } else if constexpr (MODE == 0) {
            const double f = n.b * (1.0 / TW);
            nb.a[k] = alpha * f; nb.e[k] = e * f;
            nb.eps[k] = eps; nb.w1[k] = w1;
        } else {
            nb.a[k] = alpha; nb.b[k] = n.b; nb.e[k] = e;
            nb.eps[k] = eps; nb.w1[k] = w1;
        }
    }
    __syncwarp();
    int before = -1;                                         // nodes started before the round, less one
    int k = 0;
    uint32_t en = 0;
    uint2 key = make_uint2(0u, 0u);
    auto locate = [&](int base) {                            // the lane's node and table entry of round `base`
        const unsigned m = __reduce_or_sync(FULL, act && (start >> 5) == (base >> 5) ? 1u << (start & 31) : 0u);
        k = before + __popc(m & (lt | (1u << lane)));
        before += __popc(m);
        if (base + lane < total) {
            key = nb.key[k];
            en = __ldg(tent + (uint32_t)(key.x + (uint32_t)(base + lane)));
        }
    };
    if (total > 0) locate(0);
    for (int base = 0; base < total; base += 32) {
        const int kc = k;
        const uint32_t ec = en, pk = key.y;
        if (base + 32 < total) locate(base + 32);
        if (base + lane >= total) continue;
        const int ray = (int)(ec >> 16);
        if constexpr (CD) {
            const double wk = (double)(ec & 0xffffu) * (1.0 / TW);
            atomicAdd(bins.a + ray, wk * reinterpret_cast<const double*>(&nb.w[0][0])[kc]);
            continue;
        }
        const int npts = (int)(pk >> 7) & 0xff, src = (int)(pk >> 15) & 31;
        const int b0 = ray * nr + (int)(pk & 0x7fu);
        const real* wc = &nb.w[0][src];
        if constexpr (MODE == 0) {
            const double c = widen_normal((float)(ec & 0xffffu));
            const double ca = c * nb.a[kc], ce = use_e ? c * nb.e[kc] : 0.0;
            const double d = wc[0], hpar = wc[32];
            for (int j = 0; j < npts; ++j) {
                const double w = (pk & PK_LONG)
                                     ? radial_w<double>(fabs(radius_at<double>((int)(pk & 0x7fu) + j, a.r_coef, a.r) - d), hpar, VAR ? a.kern_a : 0)
                                     : wc[j * 32];
                if (positive(ca)) atomicAdd(bins.a + b0 + j, w * ca);
                if (use_e && nonzero(ce)) atomicAdd(bins.e + b0 + j, w * ce);   // (with its sign: e is the caller's)
            }
        } else {
            // ((W b) cnt) (alpha scale / TW): the scales are powers of two
            const float c = (float)(ec & 0xffffu), b = nb.b[kc];
            const float al = nb.a[kc] * (sc.a * (1.f / TW)), ee = use_e ? nb.e[kc] * (sc.e * (1.f / TW)) : 0.f;
            double* ba = bins.a + b0;
            double* be = bins.e + b0;
            if (!(pk & PK_LONG)) {
                for (int j = 0; j < npts; ++j) {
                    const float w = wc[j * 32] * b * c;
                    bin_add_units(ba + j, w * al);
                    if (use_e) bin_add_units(be + j, w * ee);
                }
            } else {
                const float d = wc[0], hpar = wc[32];
                for (int j = 0; j < npts; ++j) {
                    const float w = radial_w<float>(fabsf(radius_at<float>((int)(pk & 0x7fu) + j, a.r_coeff, a.r) - d),
                                                    hpar, VAR ? a.kern_a : 0) * b * c;
                    bin_add_units(ba + j, w * al);
                    if (use_e) bin_add_units(be + j, w * ee);
                }
            }
        }
        if (pk & PK_EPS) {
            const real wk = (real)(ec & 0xffffu) * (real(1) / TW);
            const real ep = nb.eps[kc], s1 = nb.w1[kc], s0 = real(1) - s1;
            double* be = bins.eps + ray * nr + ((int)(pk >> 20) & 0x7f);
            if (s0 != real(0)) bin_atomic_add<MODE>(be, wk * s0 * ep, sc.eps);
            if (s1 != real(0)) bin_atomic_add<MODE>(be + 1, wk * s1 * ep, sc.eps);
        }
    }
    __syncwarp();                                            // the batch read before the next one is written
}

// The list of accepted nodes waiting to be spread: 4 NT entries, spread when
// a step could overflow it (three full batches of 32 per warp) and at the end.
// SLIM: 2 NT, spread one batch per warp at a time.
template <int NT, bool SLIM> constexpr int acc_cap() { return (SLIM ? 2 : 4) * NT; }

// Opened nodes waiting in a target's ring buffer.  While at most FIFO_MAX
// wait, the oldest are taken first, so that the list fills level by level and
// a batch of 32 accepted nodes has like numbers of points and rays; beyond
// that the newest (a depth-first walk, which bounds the buffer).  A step takes
// no more parents than the room left can hold the children of (7 more than it
// takes out each), less STACK_RESERVE: where that leaves none, one parent at a
// time, which needs at most 7 places for each of the levels 2 to 8 below it.
// So the buffer holds any walk of up to 10 levels, at any opening angle and CTA
// size (128^3 with e at theta 0.1: 589 places without the bound and 256
// threads); overflow is still detected and reported, never written past.
constexpr int STACK_CAP = 512;
constexpr int FIFO_MAX = 64;
constexpr int STACK_RESERVE = 7 * (MAX_LEVELS - 1);

// The limit on a target's ray bins and node buffer: what these leave of a CTA's
// shared memory.  Fixed figures, so that the calls that are refused do not
// change with the kernels; the smallest CTA fits beside the largest bins
// (asserted in walk_body), the larger ones where there is room.
constexpr size_t OWN_SMEM_F32 = 19072, OWN_SMEM_F64 = 40512;

// A CTA of NT threads per target.  Walk step: take NT/8 opened nodes from the
// shared buffer, evaluate their NT children, one per thread; opened children
// go back into the buffer, accepted ones with something to map to a list.  When
// the list is full, and at the end, the warps spread it (spread_nodes), 32
// nodes a warp at a time, so that two barriers a step only separate short,
// even work.  Bound by instruction issue and latency at 20 warps per SM (33
// KB of bins per target); DRAM carries the tree once.  Setting up and
// spreading the nodes of each step as they were accepted, as this walk did
// before, left a third of the lanes idle and took turbulent128 from 217 to
// 328 ms in the double-FP32 form (99 k to 62 k warp instructions per target
// in the headline form).
template <int MODE, int OUT, int NT, bool VAR, int W, bool SLIM>
__device__ __forceinline__ void walk_body(const WalkArgs* __restrict__ jobs, const int64_t* __restrict__ job_end,
                                          int n_jobs, unsigned int* counter) {
    using real = typename Prec<MODE>::real;
    constexpr int NW = NT / 32, P = NT / 8;
    constexpr bool DUMP = OUT == OUT_DUMP, CD = OUT == OUT_CD;
    extern __shared__ __align__(16) unsigned char smem[];
    // per step: stack pushes (low half) and list entries (high half),
    // reserved by one atomic per warp; two sets, by step parity, so that a
    // set is cleared a step after its use
    __shared__ unsigned s_cnt[2];
    __shared__ int s_over;
    __shared__ double s_red[NW];
    __shared__ unsigned int s_q;
    __shared__ int s_j;
    __shared__ int s_nacc;
    __shared__ __align__(16) WalkArgs s_a;                       // the current job
    __shared__ NodeBatch<MODE, W> s_nb[NW];
    __shared__ uint32_t s_acc[acc_cap<NT, SLIM>()];
    constexpr size_t own = sizeof s_nb + sizeof s_acc + sizeof s_a + sizeof s_red + 32;
    static_assert(NT != 128 || own <= (MODE == 0 ? OWN_SMEM_F64 : OWN_SMEM_F32), "the largest bins leave room for this CTA");
    // (228 KB an SM, 1 KB of it the system's per CTA; 48 rays of 59 points, alpha and eps)
    static_assert(MODE == 0 || NT != 128 || W > 7 || own <= 228 * 1024 / 4 - 1024 - 48 * 59 * 16 - STACK_CAP * 4,
                  "four targets of a 256^3 grid fit an SM");
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const WalkArgs& a = s_a;
    const unsigned lanemask_lt = (1u << lane) - 1u;
    const int64_t total = job_end[n_jobs - 1];
    WalkCounters cnt;                                        // per-thread counters
    float kap = 0.f;                                         // FP32 forms: the tree's kappa
    int cur = -1;
    unsigned done = 0;                                       // targets since the counters were flushed
    int nr = 0, nbins = 0, nq = 2, N = 0, L = 0;
    Scales sc{1.f, 1.f, 1.f};

    for (;;) {
        if (tid == 0) {
            const unsigned int qq = atomicAdd(counter, 1u);
            int j = -1;
            if ((int64_t)qq < total) { j = 0; while (job_end[j] <= (int64_t)qq) ++j; }
            s_q = qq;
            s_j = j;
        }
        __syncthreads();
        const int j = s_j;
        const int64_t qg = (int64_t)s_q;
        if (j < 0) break;
        if (cur >= 0 && (j != cur || ++done >= FLUSH_TARGETS)) { flush_counters(a, cnt); done = 0; }
        if (j != cur) {                                          // load the job (uniform over the CTA)
            __syncthreads();
            const int* src = reinterpret_cast<const int*>(jobs + j);
            int* dst = reinterpret_cast<int*>(&s_a);
            for (int k = tid; k < (int)(sizeof(WalkArgs) / sizeof(int)); k += NT) dst[k] = src[k];
            __syncthreads();
            cur = j;
            nr = a.nr; nbins = CD ? a.npix : a.npix * nr; nq = CD ? 1 : (a.use_e ? 3 : 2); N = a.N; L = a.L;
            if (MODE != 0) {                                     // fixed-point units from the root totals
                real cm0[3], m0, q0[3], mi0;
                load_node<MODE>(a.nodes, 0, cm0, m0, q0, mi0);
                sc.a = fixed_scale((float)q0[0]);
                sc.eps = fixed_scale((float)q0[1]);
                sc.e = fixed_scale((float)q0[2]);
                kap = __ldg(a.kappa) * 1.000001f;
            }
        }
        // derived from smem here, unconditionally, so that they stay shared-memory
        // pointers to the compiler (a null on some path makes them generic)
        double* const bins_a = reinterpret_cast<double*>(smem);
        const Bins bins{bins_a, bins_a + nbins, bins_a + 2 * nbins};
        uint32_t* const stack = reinterpret_cast<uint32_t*>(bins_a + nq * nbins);
        const int64_t q = qg - (j > 0 ? job_end[j - 1] : 0);    // index within the job
        if (a.targets) {                                         // caller's list: reject bad indices
            const int64_t c = a.targets[q];
            if (c < 0 || c >= a.n_cells) {                       // (uniform over the CTA)
                if (tid == 0) atomicAdd(a.status + 2, 1);
                __syncthreads();                                 // s_q, s_j read before thread 0 rewrites them
                continue;
            }
        }
        Target<MODE> t;
        t.ts = 1;
        int tl = L;                                              // the target's level
        int64_t cell;
        if (a.blk) {                                             // AMR: cell c of block b
            int b, lx, ly, lz;
            if (a.targets) {
                cell = a.targets[q];
                b = (int)(cell >> 9);
                const int c = (int)(cell & 511);
                lx = c & 7; ly = (c >> 3) & 7; lz = c >> 6;
            } else {
                const int64_t k = a.first + q;
                b = (int)__ldg(a.blk_order + (k >> 9));
                const uint32_t lm = (uint32_t)(k & 511);
                lx = (int)compact3(lm); ly = (int)compact3(lm >> 1); lz = (int)compact3(lm >> 2);
                cell = ((int64_t)b << 9) + (lz * 8 + ly) * 8 + lx;
            }
            const int4 bm = __ldg(a.blk + b);
            tl = bm.x;
            t.ts = N >> tl;
            t.tx = (8 * bm.y + lx) * t.ts; t.ty = (8 * bm.z + ly) * t.ts; t.tz = (8 * bm.w + lz) * t.ts;
        } else if (a.targets) {
            cell = a.targets[q];
            t.tx = (int)(cell % N); t.ty = (int)((cell / N) % N); t.tz = (int)(cell / ((int64_t)N * N));
        } else {
            const uint32_t m = (uint32_t)(a.first + q);
            t.tx = (int)compact3(m); t.ty = (int)compact3(m >> 1); t.tz = (int)compact3(m >> 2);
            cell = ((int64_t)t.tz * N + t.ty) * N + t.tx;
        }
        const real hts = real(0.5) * (real)t.ts;
        t.px = (real)t.tx + hts; t.py = (real)t.ty + hts; t.pz = (real)t.tz + hts;
        // (npix and so nbins is a multiple of 12)
        for (int b = tid; b < nq * nbins / 2; b += NT) reinterpret_cast<double2*>(bins_a)[b] = make_double2(0.0, 0.0);
        if (tid == 0) {                                          // the root, opened
            stack[0] = 0u; s_nacc = 0;
            s_cnt[0] = s_cnt[1] = 0u; s_over = 0;
        }
        int head = 0, top = 1, max_top = 1, par = 0, nl = 0;     // top: waiting nodes (from head on); nl: listed nodes
        bool overflow = false;
        __syncthreads();
        // spread the last `take` listed nodes, 32 per warp at a time
        auto spread_list = [&](int take, int img) {
            if constexpr (CD) {
                // every node deposits on few rays and siblings on the same ones:
                // a batch of nodes from all over the list retries fewer FP64
                // atomics (64^3: 20.7 -> 16.4 ms)
                const int batches = (take + 31) >> 5;
                for (int b = wid; b < batches; b += NW) {
                    const int k = nl - take + b + lane * batches;
                    const bool have = k < nl;
                    spread_nodes<MODE, OUT, VAR>(a, s_nb[wid], have ? s_acc[k] : 0u, have, img, t, bins, sc, kap, cnt);
                }
            } else {
                for (int b = nl - take + wid * 32; b < nl; b += NT) {
                    const bool have = b + lane < nl;
                    spread_nodes<MODE, OUT, VAR>(a, s_nb[wid], have ? s_acc[b + lane] : 0u, have, img, t, bins, sc, kap, cnt);
                }
            }
            nl -= take;
        };
        // corner of symmetry: the original and its 7 mirror images (bit k of
        // img mirrors axis k through the low corner), all onto the same rays
        const int n_img = (VAR && a.bc == TR_BC_CORNER) ? 8 : 1;
        for (int img = 0; img < n_img && !overflow; ++img) {
        if (img > 0) {
            if (tid == 0) stack[head & (STACK_CAP - 1)] = ROOT_EVAL;
            top = 1;
            __syncthreads();                                     // the image's root visible, the list read
        }
        for (;;) {
            if (top == 0 || nl + NT > acc_cap<NT, SLIM>()) {           // the walk's end, or a full list: full batches
                spread_list(top == 0 ? nl : nl / NT * NT, img);
                if (top == 0) break;
            }
            int np = min(P, top);
            if (top > STACK_CAP - STACK_RESERVE - 7 * P) np = max(min(np, (STACK_CAP - STACK_RESERVE - top) / 7), 1);
            const int pi = tid >> 3, c = tid & 7;
            const bool fifo = top <= FIFO_MAX;
            const uint32_t pe = (pi < np) ? stack[(head + (fifo ? 0 : top - np) + pi) & (STACK_CAP - 1)] : 0u;
            __syncthreads();                                     // parents and list read before they are overwritten
            top -= np;
            if (fifo) head += np;
            int action = 0;                                      // 1 open, 2 accept
            uint32_t ent = 0;                                    // the child as a stack or list entry
            bool list = false;
            // ROOT_EVAL: the root itself is evaluated (a mirror image does not
            // contain the target, so its root is subject to the MACs)
            if (pi < np && (!VAR || pe != ROOT_EVAL || c == 0)) {
                ++cnt.vis;
                const int lev = (VAR && pe == ROOT_EVAL) ? 0 : (int)(pe >> 27) + 1;
                const uint32_t mort = (VAR && pe == ROOT_EVAL) ? 0u : (((pe & 0x7ffffffu) << 3) | (uint32_t)c);
                ent = ((uint32_t)lev << 27) | mort;
                const int s = N >> lev;
                const int cx = (int)compact3(mort) * s, cy = (int)compact3(mort >> 1) * s,
                          cz = (int)compact3(mort >> 2) * s;
                const bool contains = img == 0 && (t.tx >= cx && t.tx < cx + s) && (t.ty >= cy && t.ty < cy + s) &&
                                      (t.tz >= cz && t.tz < cz + s);
                const int64_t nid = level_offset(lev) + mort;
                const bool leaf = a.flags ? (__ldg(a.flags + nid) == NODE_LEAF) : (lev == L);
                if (contains) {
                    action = leaf ? 0 : 1;                       // a leaf holding the target is the target
                } else {
                    real cm[3], m, qv[3], mion;
                    load_node<MODE>(a.nodes, nid, cm, m, qv, mion);
                    bool open = false;
                    if (!leaf) {
                        const NodeView<MODE> v = view_node<MODE, VAR>(a, t, img, cx, cy, cz, s, cm, kap);
                        const real h2 = (real)s * (real)s;
                        if constexpr (MODE == 0) {
                            open = must_open(h2, v.d2, m, mion, qv[1], a);
                        } else {
                            const int r = mac_f32(h2, v.d2, v.B, signbit(mion), qv[1] > 0.f, a);
                            if (r < 0) {
                                ++cnt.fb_mac;
                                open = must_open_exact((double)h2, exact_d2(a, nid, v.qx, v.qy, v.qz), signbit(mion),
                                                       qv[1] > 0.f, a);
                            } else {
                                open = r == 1;
                            }
                        }
                    }
                    action = open ? 1 : 2;
                    list = !open && (CD ? m > real(0)
                                        : (qv[0] != real(0) || qv[1] != real(0) || (a.use_e && qv[2] != real(0))));
                }
            }
            // slots of the pushes and of the listed nodes: one shared atomic
            // per warp reserves both (the order of the warps' blocks is
            // immaterial: fixed-point or FP64 atomic deposits, accepted
            // nodes a set)
            const unsigned om = __ballot_sync(FULL, action == 1);
            const unsigned bm = __ballot_sync(FULL, list);
            unsigned base = 0;
            if (lane == 0 && (om | bm)) base = atomicAdd(&s_cnt[par], ((unsigned)__popc(bm) << 16) | (unsigned)__popc(om));
            base = __shfl_sync(FULL, base, 0);
            if (action == 1) {
                const int slot = top + (int)(base & 0xffffu) + __popc(om & lanemask_lt);
                if (slot < STACK_CAP) stack[(head + slot) & (STACK_CAP - 1)] = ent;
                else s_over = 1;                                 // never written past
            }
            if (list) s_acc[nl + (int)(base >> 16) + __popc(bm & lanemask_lt)] = ent;   // nl + NT <= acc_cap
            if (action == 2) {
                ++cnt.acc;
                if (DUMP) {
                    const int slot = atomicAdd(&s_nacc, 1);
                    if (slot < a.acc_cap) a.ids_out[q * a.acc_cap + slot] = (int32_t)(level_offset((int)(ent >> 27)) + (ent & 0x7ffffffu));
                }
            }
            __syncthreads();                                     // pushes and list visible
            const unsigned added = s_cnt[par];
            overflow = s_over != 0;                              // same value in every thread
            if (tid == 0) s_cnt[par ^ 1] = 0u;                   // read by all a step ago
            par ^= 1;
            if (overflow) break;
            top += (int)(added & 0xffffu);
            nl += (int)(added >> 16);
            max_top = max(max_top, top);
        }
        }                                                        // images
        __syncthreads();                                         // all spreads done
        if (CD) {
            if (tid == 0) atomicMax(a.status + 1, max_top);
            if (overflow) {
                if (tid == 0) atomicAdd(a.status, 1);
                continue;
            }
            double* out = a.cd_out + (size_t)(a.targets ? q : cell) * a.npix;
            for (int k = tid; k < a.npix; k += NT) out[k] = bins.a[k] * a.cd_conv;
            continue;
        }
        // own emission of the target (Sec. 2.5 footnote: target sphere of
        // radius r_tp = half the cell edge)
        real cmt[3], mt, qt[3], miont;
        load_node<MODE>(a.nodes, level_offset(tl) + morton3(t.tx / t.ts, t.ty / t.ts, t.tz / t.ts), cmt, mt, qt, miont);
        const double r_tp2 = 0.25 * (double)t.ts * (double)t.ts;
        const double eps_self = (double)qt[1];
        if (tid == 0) atomicMax(a.status + 1, max_top);
        if (overflow) {
            if (tid == 0) {
                atomicAdd(a.status, 1);
                if (a.F) a.F[a.targets ? q : cell] = __longlong_as_double(0x7ff8000000000000LL);
            }
            continue;
        }
        if (DUMP) {                                              // raw bins, as the sweep reads them
            double* out = a.bins_out + (size_t)q * 3 * nbins;
            for (int b = tid; b < nbins; b += NT) {
                out[b] = bins.a[b];
                out[nbins + b] = bins.eps[b];
                out[2 * nbins + b] = a.use_e ? bins.e[b] : 0.0;
            }
            if (tid == 0) {
                a.counts_out[q] = s_nacc;
                a.eps_self_out[q] = eps_self / ((double)t.ts * (double)t.ts);   // reaches the centre as for ts = 1
                if (q == 0) { a.scales_out[0] = sc.a; a.scales_out[1] = sc.eps; a.scales_out[2] = sc.e; }
            }
            continue;
        }
        const int turn = MODE == 2 ? 0 : (int)q;
        static_assert(sizeof s_nb >= sweep_scratch_bytes(MAX_NPIX, 64) && sizeof s_nb >= sweep_scratch_bytes(192, MAX_NR),
                      "the sweep's tables fit the spread's memory");
        const double Fk = sweep_rays<MODE, NT>(a, bins.a, bins.eps, bins.e, sc, reinterpret_cast<unsigned char*>(s_nb), turn);
        const double F = block_sum<NT>(Fk, s_red, turn) + eps_self / (4.0 * PI_D * r_tp2);
        if (tid == 0) {
            const int64_t o = a.targets ? q : cell;
            if (a.F) a.F[o] = F * a.Fconv;
            if (a.E) a.E[o] = F * a.Econv;
            if (a.ion) a.ion[o] = (uint8_t)(F > 0.0);
        }
    }
    if (cur >= 0) flush_counters(a, cnt);
}

// CTAS: the CTAs per SM that the registers have to allow.
template <int MODE, int OUT, int NT, int CTAS, bool VAR, bool SLIM = false>
__global__ void __launch_bounds__(NT, CTAS) k_walk(const WalkArgs* __restrict__ jobs, const int64_t* __restrict__ job_end,
                                                  int n_jobs, unsigned int* counter) {
    walk_body<MODE, OUT, NT, VAR, MAXW<MODE, NT, CTAS, VAR, SLIM>, SLIM>(jobs, job_end, n_jobs, counter);
}

// Unfused sweep over bins stored by the dump walk: one CTA per target.
template <int MODE, int NT>
__global__ void __launch_bounds__(NT) k_sweep_stored(WalkArgs a, const double* bins_in, const double* eps_self) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_red[NT / 32];
    const int tid = threadIdx.x;
    const int nbins = a.npix * a.nr;
    double* bins_a = reinterpret_cast<double*>(smem);
    double* bins_eps = bins_a + nbins;
    double* bins_e = a.use_e ? bins_eps + nbins : nullptr;
    for (int64_t q = blockIdx.x; q < a.n_targets; q += gridDim.x) {
        const double* in = bins_in + (size_t)q * 3 * nbins;
        __syncthreads();
        for (int b = tid; b < nbins; b += NT) {
            bins_a[b] = in[b];
            bins_eps[b] = in[nbins + b];
            if (a.use_e) bins_e[b] = in[2 * nbins + b];
        }
        __syncthreads();
        const int turn = MODE == 2 ? 0 : (int)q;
        const double Fk = sweep_rays<MODE, NT>(a, bins_a, bins_eps, bins_e,
                                               Scales{a.scales_in[0], a.scales_in[1], a.scales_in[2]},
                                               smem + (size_t)(a.use_e ? 3 : 2) * nbins * sizeof(double), turn);
        const double F = block_sum<NT>(Fk, s_red, turn) + eps_self[q] / (4.0 * PI_D * 0.25);
        if (tid == 0) {
            if (a.F) a.F[q] = F * a.Fconv;
            if (a.E) a.E[q] = F * a.Econv;
            if (a.ion) a.ion[q] = (uint8_t)(F > 0.0);
        }
    }
}

constexpr int SWEEP_NT = 128;               // threads per target of the stored-bins sweep

// Before a walk of one tree: its job record (passed as the kernel's parameter,
// so that no host buffer has to outlive the call), its status words and
// counters cleared, and the work counter.  One launch in place of three
// clears, a copy and a wait for the copy (16^3 solve 281 -> 267 us).
__global__ void __launch_bounds__(128) k_job_start(const __grid_constant__ WalkArgs a, int64_t end, WalkArgs* job, int64_t* job_end,
                                                   unsigned int* counter) {
    const int* src = reinterpret_cast<const int*>(&a);
    for (int k = threadIdx.x; k < (int)(sizeof(WalkArgs) / sizeof(int)); k += 128) reinterpret_cast<int*>(job)[k] = src[k];
    if (threadIdx.x < 4) a.status[threadIdx.x] = 0;
    if (threadIdx.x < N_STATS) a.stats[threadIdx.x] = 0ull;
    if (threadIdx.x == 0) { *job_end = end; *counter = 0u; }
}

tr_status job_start(const WalkArgs& a, const tr_tree* t, int64_t n_targets, const WalkArgs** jobs, const int64_t** job_end,
                    cudaStream_t st) {
    WalkArgs* j = reinterpret_cast<WalkArgs*>(t->jobbuf);
    int64_t* e = reinterpret_cast<int64_t*>(reinterpret_cast<unsigned char*>(t->jobbuf) + sizeof(WalkArgs));
    k_job_start<<<1, 128, 0, st>>>(a, n_targets, j, e, t->counter);
    *jobs = j;
    *job_end = e;
    return cuda_check(cudaGetLastError(), "job record kernel");
}

size_t walk_smem(const tr_tree* t) {
    const int nq = t->use_e ? 3 : 2;
    return (size_t)nq * t->npix * t->nr * 8 + (size_t)STACK_CAP * 4;
}

WalkArgs make_args(const tr_tree* t) {
    WalkArgs a{};
    a.nodes = t->nodes;
    a.nodes64 = (const NodeF64*)t->nodes64;
    a.kappa = t->kappa;
    a.N = t->N; a.L = t->L; a.nr = t->nr; a.npix = t->npix; a.eta = t->p.eta_r; a.nside = t->p.nside;
    a.use_e = t->use_e;
    a.th_lim2 = t->p.theta_lim * t->p.theta_lim;
    a.th_if2 = t->p.theta_if * t->p.theta_if;
    a.th_src2 = t->p.theta_src * t->p.theta_src;
    a.lray = t->lray;
    a.r_coef = 1.0 / (2.0 * (double)t->p.eta_r * (double)t->p.eta_r);
    a.r_coeff = (float)a.r_coef;
    a.th_lim2f = (float)a.th_lim2; a.th_if2f = (float)a.th_if2; a.th_src2f = (float)a.th_src2;
    a.lrayf = (float)t->lray;
    a.toff = t->table->off; a.tent = t->table->ent; a.hdr = t->table->hdr;
    a.r = t->sw.r; a.rf = t->sw.rf; a.inv_r2 = t->sw.inv_r2; a.inv_vol = t->sw.inv_vol; a.inv_volf = t->sw.inv_volf;
    a.ID2 = t->sw.ID2; a.GI = t->sw.GI; a.Gf = t->sw.Gf; a.ID2f = t->sw.ID2f; a.GIf = t->sw.GIf;
    a.HT = t->sw.HT;
    a.Fconv = t->U / (t->dx * t->dx);
    a.Econv = t->Eu;
    a.status = t->status;
    a.stats = t->stats;
    a.n_cells = t->n_cells;
    a.kern_a = t->p.kernel_alpha;
    a.kern_e = t->p.kernel_eps;
    a.bc = t->p.bc;
    a.flags = t->flags;
    a.blk = t->blk;
    a.blk_order = t->blk_order;
    return a;
}

// A kernel's limit on dynamic shared memory is one value for all threads of the
// process; it is set for each launch and each query of a fit, so both hold this
// lock from there on.
std::mutex g_smem_limit_mu;

template <int NT, typename K>
tr_status launch_persistent(K kernel, size_t smem, const WalkArgs* jobs, const int64_t* job_end, int n_jobs,
                            int64_t total, unsigned int* counter, cudaStream_t st) {
    std::lock_guard<std::mutex> lock(g_smem_limit_mu);
    tr_status s = cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                             "cudaFuncSetAttribute(smem)");
    if (s != TR_OK) return s;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    s = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, NT, smem), "occupancy query");
    if (s != TR_OK) return s;
    if (per_sm < 1) return set_error(TR_EUNSUPPORTED, "ray bins need %zu bytes of shared memory per target", smem);
    int64_t blocks = (int64_t)sms * per_sm;
    if (blocks > total) blocks = total > 0 ? total : 1;
    kernel<<<(unsigned)blocks, NT, smem, st>>>(jobs, job_end, n_jobs, counter);
    return cuda_check(cudaGetLastError(), "walk kernel launch");
}

// CTAs that one SM holds of a walk kernel with `smem` bytes of bins and
// buffer (0: it does not fit).
template <int NT, typename K>
int resident_ctas(K kernel, size_t smem) {
    int per_sm = 0;
    std::lock_guard<std::mutex> lock(g_smem_limit_mu);
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, NT, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return per_sm;
}

// The CTA of a walk: 128 threads with registers for five (K5) or six (K6) on an
// SM, 256 or 512 threads; 512 with less memory of its own; and the CTAs that an
// SM then holds.
enum CtaKind { K5, K6, K256, K512, K512_SLIM };
struct CtaPick { CtaKind kind = K5; int per_sm = 0; };

// The ray bins' shared memory sets how many targets an SM holds.  Small CTAs
// hold more of them; large ones bring more warps to each.  A target's sweep by
// lane pairs keeps 2 N_PIX threads busy whatever the CTA has, so the fused walk
// takes the CTA with the most threads on an SM that sweep, the most warps
// among equals (the walk waits on memory and its barriers), the smaller CTA
// among equals again.  Measured, FP32 + FP64-sweep form, ms:
//   N_PIX 48, 256^3, 100 sources, 2^20 targets: 4 x 128 329, 2 x 256 515
//   N_PIX 48, 128^3 with e, 10^3 sources, 2^18: 3 x 128  91, 2 x 256 112
//   N_PIX 48, 256^3 with e, 100 sources, 2^20:  2 x 128 710, 2 x 256 619
//   N_PIX 192, 64^3, 10^3 sources, 2^17:        2 x 128  58, 2 x 256  42, 1 x 512 61
//   N_PIX 192, 64^3 with e, 10^3 sources, 2^16: 1 x 128  69, 1 x 256  46, 1 x 512 39
// The most warps alone, the rule before, took 2 x 256 in the first two, and the
// many-source walks of 256^3 grids were slower than with 4 x 128 smaller steps.
// The slim 512-thread CTA (31 KB of its own instead of 37) is for bins that
// leave the other no room, as 128^3 grids with e at N_PIX 192 do (double-FP32
// form, 10^3 sources, 2^16 targets: 256 threads 73 ms, slim 50 ms); where both
// fit it is 2 to 10% slower.  The dump walk does not sweep: most warps.  MODE 2
// (double-FP32 sweep) only differs from MODE 1 in the sweep, so its dump and
// column-density walks are those of MODE 1 (chosen by launch_jobs).
template <int MODE, int OUT, bool VAR>
CtaPick pick_cta(size_t smem, int npix) {
    CtaPick best;
    int lanes = -1, warps = -1;
    auto consider = [&](CtaKind kind, int nt, int per_sm) {
        const int w = per_sm * nt / 32, l = OUT == OUT_FUSED ? per_sm * std::min(nt, 2 * npix) : w;
        if (l > lanes || (l == lanes && w > warps)) {
            best = {kind, per_sm};
            lanes = l;
            warps = w;
        }
    };
    consider(K5, 128, resident_ctas<128>(k_walk<MODE, OUT, 128, 5, VAR>, smem));
    if constexpr (OUT == OUT_FUSED && MODE != 0) consider(K6, 128, resident_ctas<128>(k_walk<MODE, OUT, 128, 6, VAR>, smem));
    // (registers allow two CTAs of 256 threads and one of 512: not asked where that cannot win)
    auto worth = [&](int nt, int per_sm) { return OUT != OUT_FUSED || per_sm * std::min(nt, 2 * npix) >= lanes; };
    if (worth(256, 2)) consider(K256, 256, resident_ctas<256>(k_walk<MODE, OUT, 256, 2, VAR>, smem));
    if constexpr (MODE != 0)
        if (worth(512, 1)) {
            const int n = resident_ctas<512>(k_walk<MODE, OUT, 512, 1, VAR>, smem);
            consider(K512, 512, n);
            if constexpr (OUT == OUT_FUSED)
                if (n == 0) consider(K512_SLIM, 512, resident_ctas<512>(k_walk<MODE, OUT, 512, 1, VAR, true>, smem));
        }
    return best;
}

// Ray bins of a launch: the most bytes (with the node buffer) and the most rays
// of any of its targets.
struct BinShape { size_t smem; int npix; };

template <int MODE, int OUT, bool VAR>
tr_status launch_sized(BinShape b, const WalkArgs* jobs, const int64_t* job_end, int n_jobs, int64_t total,
                       unsigned int* counter, cudaStream_t st) {
    auto* const k5 = k_walk<MODE, OUT, 128, 5, VAR>;
    if constexpr (OUT != OUT_CD) {                            // (column densities: few bins, 128 threads always)
        const CtaKind kind = pick_cta<MODE, OUT, VAR>(b.smem, b.npix).kind;
        if constexpr (OUT == OUT_FUSED && MODE != 0)
            if (kind == K6) return launch_persistent<128>(k_walk<MODE, OUT, 128, 6, VAR>, b.smem, jobs, job_end, n_jobs, total, counter, st);
        if constexpr (OUT == OUT_FUSED && MODE != 0)
            if (kind == K512_SLIM) return launch_persistent<512>(k_walk<MODE, OUT, 512, 1, VAR, true>, b.smem, jobs, job_end, n_jobs, total, counter, st);
        if constexpr (MODE != 0)
            if (kind == K512) return launch_persistent<512>(k_walk<MODE, OUT, 512, 1, VAR>, b.smem, jobs, job_end, n_jobs, total, counter, st);
        if (kind == K256) return launch_persistent<256>(k_walk<MODE, OUT, 256, 2, VAR>, b.smem, jobs, job_end, n_jobs, total, counter, st);
    }
    return launch_persistent<128>(k5, b.smem, jobs, job_end, n_jobs, total, counter, st);
}

template <int MODE, bool VAR>
tr_status launch_mode(int out, BinShape b, const WalkArgs* jobs, const int64_t* job_end, int n_jobs, int64_t total,
                      unsigned int* counter, cudaStream_t st) {
    if constexpr (MODE != 2) {
        if (out == OUT_CD) return launch_sized<MODE, OUT_CD, VAR>(b, jobs, job_end, n_jobs, total, counter, st);
        if (out == OUT_DUMP) return launch_sized<MODE, OUT_DUMP, VAR>(b, jobs, job_end, n_jobs, total, counter, st);
    }
    return launch_sized<MODE, OUT_FUSED, VAR>(b, jobs, job_end, n_jobs, total, counter, st);
}

template <bool VAR>
tr_status launch_jobs_v(int mode, int out, BinShape b, const WalkArgs* jobs, const int64_t* job_end,
                        int n_jobs, int64_t total, unsigned int* counter, cudaStream_t st) {
    if (mode == 0) return launch_mode<0, VAR>(out, b, jobs, job_end, n_jobs, total, counter, st);
    if (mode == 1 || out != OUT_FUSED)
        return launch_mode<1, VAR>(out, b, jobs, job_end, n_jobs, total, counter, st);
    return launch_mode<2, VAR>(out, b, jobs, job_end, n_jobs, total, counter, st);
}

// The one refusal of a walk: bins that no CTA can hold.
tr_status check_bins(int mode, int out, size_t smem) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    tr_status c = cuda_check(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev),
                             "shared memory limit");
    if (c != TR_OK) return c;
    const size_t own = out == OUT_CD ? 0 : (mode == 0 ? OWN_SMEM_F64 : OWN_SMEM_F32);
    if (smem + own > (size_t)optin)
        return set_error(TR_EUNSUPPORTED,
                         "ray bins need %zu + %zu bytes of shared memory per target, more than the %d a CTA can have"
                         " (fewer rays, a shorter L_ray or no e_prev)", smem, own, optin);
    return TR_OK;
}

// var: some job uses a kernel choice other than W_p / W_f,3 or a boundary
// other than isolated
tr_status launch_jobs(int mode, int out, bool var, BinShape b, const WalkArgs* jobs, const int64_t* job_end,
                      int n_jobs, int64_t total, unsigned int* counter, cudaStream_t st) {
    const tr_status c = check_bins(mode, out, b.smem);
    if (c != TR_OK) return c;
    return var ? launch_jobs_v<true>(mode, out, b, jobs, job_end, n_jobs, total, counter, st)
               : launch_jobs_v<false>(mode, out, b, jobs, job_end, n_jobs, total, counter, st);
}

// Targets that an SM holds at once in the fused walk of a form.
template <bool VAR>
int targets_per_sm(int mode, BinShape b) {
    return (mode == 0 ? pick_cta<0, OUT_FUSED, VAR>(b.smem, b.npix)
            : mode == 1 ? pick_cta<1, OUT_FUSED, VAR>(b.smem, b.npix) : pick_cta<2, OUT_FUSED, VAR>(b.smem, b.npix)).per_sm;
}
// Targets per resident target below which a batch's group is too small to launch
// alone.  0 to 16 measured the same on seven batches of two to nine trees (16^3 to
// 128^3, N_PIX 48 and 192, a slice of 256^3), one launch for all 3 to 90% slower.
constexpr int BATCH_WAVES = 4;

bool uses_variants(const tr_tree* t) {
    return t->p.kernel_alpha != TR_KERNEL_WP || t->p.kernel_eps != TR_EPS_WF3 || t->p.bc != TR_BC_ISOLATED;
}

}  // namespace

size_t walk_job_bytes(int n_jobs) { return (size_t)n_jobs * (sizeof(WalkArgs) + sizeof(int64_t)); }

tr_status walk_run(const tr_tree* t, const int64_t* targets, int64_t n_targets, bool dump, const WalkOut& out,
                   cudaStream_t st) {
    WalkArgs a = make_args(t);
    a.targets = targets;
    a.first = 0;
    a.n_targets = n_targets;
    a.F = out.F; a.E = out.e; a.ion = out.ion;
    a.bins_out = out.bins; a.ids_out = out.ids; a.counts_out = out.counts; a.eps_self_out = out.eps_self;
    a.scales_out = out.scales;
    a.acc_cap = out.acc_cap;
    const WalkArgs* jobs = nullptr;
    const int64_t* job_end = nullptr;
    const tr_status s = job_start(a, t, n_targets, &jobs, &job_end, st);
    if (s != TR_OK || n_targets <= 0) return s;
    return launch_jobs(t->mode, dump ? OUT_DUMP : OUT_FUSED, uses_variants(t),
                       {walk_smem(t), t->npix}, jobs, job_end, 1, n_targets, t->counter, st);
}

tr_status cd_run(const tr_tree* t, const int64_t* targets, int64_t n_targets, double* out, cudaStream_t st) {
    WalkArgs a = make_args(t);
    a.targets = targets;
    a.first = 0;
    a.n_targets = n_targets;
    a.cd_out = out;
    a.cd_conv = t->dx;
    a.cd_omega = 4.0 * PI_D / (double)t->npix;
    const WalkArgs* jobs = nullptr;
    const int64_t* job_end = nullptr;
    const tr_status s = job_start(a, t, n_targets, &jobs, &job_end, st);
    if (s != TR_OK || n_targets <= 0) return s;
    const size_t smem = (size_t)t->npix * 8 + (size_t)STACK_CAP * 4;
    return launch_jobs(t->mode, OUT_CD, uses_variants(t), {smem, t->npix}, jobs, job_end, 1, n_targets, t->counter, st);
}

tr_status walk_batch_run(const tr_tree* const* trees, const int64_t* first, const int64_t* count, int n,
                         double* const* F, double* const* e, uint8_t* const* ion, void* jobbuf, unsigned int* counter,
                         cudaStream_t st) {
    // Jobs by the number of targets that an SM holds at once with each tree's
    // own ray bins, one launch for each: a tree with N_PIX 192 would otherwise
    // set the shared memory, and so the warps per SM, of every target (two 64^3
    // and two 32^3 trees, one with N_PIX 192: 141 -> 76 ms).  A group too small
    // to fill the GPU a few times over joins the next with larger bins.
    struct Item { int tree, per_sm; size_t smem; };
    const int mode = trees[0]->mode;
    tr_status s = TR_OK;
    // a batch with a tree that cannot be walked, an idle one too, is refused as
    // a whole, before anything is launched
    size_t largest = 0;
    bool any = false;
    for (int i = 0; i < n; ++i) {
        largest = std::max(largest, walk_smem(trees[i]));
        any = any || count[i] > 0;
    }
    if (any && (s = check_bins(mode, OUT_FUSED, largest)) != TR_OK) return s;
    std::vector<Item> items;
    for (int i = 0; i < n; ++i)
        if (count[i] > 0) {
            const size_t m = walk_smem(trees[i]);
            const BinShape b{m, trees[i]->npix};
            items.push_back({i, uses_variants(trees[i]) ? targets_per_sm<true>(mode, b) : targets_per_sm<false>(mode, b), m});
        }
    std::stable_sort(items.begin(), items.end(), [](const Item& x, const Item& y) { return x.per_sm > y.per_sm; });
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    std::vector<unsigned char> host(walk_job_bytes(n));
    WalkArgs* hj = reinterpret_cast<WalkArgs*>(host.data());
    int64_t* he = reinterpret_cast<int64_t*>(host.data() + (size_t)n * sizeof(WalkArgs));
    struct Group { int first, n; BinShape b; int64_t total; bool var; };
    std::vector<Group> groups;
    for (int k = 0; k < (int)items.size(); ++k) {
        const int i = items[k].tree;
        const bool join = k > 0 && (items[k].per_sm == items[k - 1].per_sm ||
                                    groups.back().total < (int64_t)sms * items[k - 1].per_sm * BATCH_WAVES);
        if (!join) groups.push_back({k, 0, {0, 0}, 0, false});
        Group& g = groups.back();
        WalkArgs a = make_args(trees[i]);
        a.targets = nullptr;
        a.first = first[i];
        a.n_targets = count[i];
        a.F = F ? F[i] : nullptr; a.E = e ? e[i] : nullptr; a.ion = ion ? ion[i] : nullptr;
        hj[k] = a;
        ++g.n;
        g.total += count[i];
        he[k] = g.total;
        g.b = {std::max(g.b.smem, items[k].smem), std::max(g.b.npix, trees[i]->npix)};
        g.var = g.var || uses_variants(trees[i]);
    }
    for (int i = 0; i < n; ++i) {
        if (s == TR_OK) s = cuda_check(cudaMemsetAsync(trees[i]->status, 0, 4 * sizeof(int32_t), st), "status reset");
        if (s == TR_OK) s = cuda_check(cudaMemsetAsync(trees[i]->stats, 0, N_STATS * sizeof(unsigned long long), st), "stats reset");
    }
    if (s == TR_OK) s = cuda_check(cudaMemcpyAsync(jobbuf, host.data(), host.size(), cudaMemcpyHostToDevice, st), "job copy");
    if (s == TR_OK) s = cuda_check(cudaStreamSynchronize(st), "job copy");
    const WalkArgs* jobs = reinterpret_cast<const WalkArgs*>(jobbuf);
    const int64_t* job_end = reinterpret_cast<const int64_t*>(reinterpret_cast<unsigned char*>(jobbuf) + (size_t)n * sizeof(WalkArgs));
    for (const Group& g : groups) {
        if (s == TR_OK) s = cuda_check(cudaMemsetAsync(counter, 0, sizeof(unsigned int), st), "counter reset");
        if (s == TR_OK)
            s = launch_jobs(mode, OUT_FUSED, g.var, g.b, jobs + g.first, job_end + g.first, g.n, g.total, counter, st);
    }
    // an earlier group may be running: it uses the caller's outputs and the
    // shared job records, which the caller may reuse after an error
    if (s != TR_OK) cudaStreamSynchronize(st);
    return s;
}

tr_status sweep_run(const tr_rays* r, double* F, double* e, uint8_t* ion, cudaStream_t st) {
    WalkArgs a{};
    a.nr = r->nr; a.npix = r->npix; a.use_e = r->use_e;
    a.r = r->sw.r; a.inv_r2 = r->sw.inv_r2; a.inv_vol = r->sw.inv_vol; a.inv_volf = r->sw.inv_volf; a.ID2 = r->sw.ID2; a.GI = r->sw.GI; a.Gf = r->sw.Gf; a.ID2f = r->sw.ID2f; a.GIf = r->sw.GIf;
    a.HT = r->sw.HT;
    a.n_targets = r->n_targets;
    a.Fconv = r->U / (r->dx * r->dx);
    a.Econv = r->Eu;
    a.F = F; a.E = e; a.ion = ion;
    a.scales_in = r->scales;
    const size_t smem = (size_t)(r->use_e ? 3 : 2) * r->npix * r->nr * 8 + sweep_scratch_bytes(r->npix, r->nr);
    auto kern = r->mode == 0 ? k_sweep_stored<0, SWEEP_NT>
                             : (r->mode == 1 ? k_sweep_stored<1, SWEEP_NT> : k_sweep_stored<2, SWEEP_NT>);
    std::lock_guard<std::mutex> lock(g_smem_limit_mu);
    tr_status s = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                             "cudaFuncSetAttribute(sweep smem)");
    if (s != TR_OK) return s;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t blocks = r->n_targets < (int64_t)sms * 4 ? r->n_targets : (int64_t)sms * 4;
    if (blocks > 0) kern<<<(unsigned)blocks, SWEEP_NT, smem, st>>>(a, r->bins, r->eps_self);
    return cuda_check(cudaGetLastError(), "sweep kernel launch");
}

tr_status read_status(const tr_tree* t, cudaStream_t st) {
    int32_t h[4] = {0, 0, 0, 0};
    tr_status s = cuda_check(cudaMemcpyAsync(h, t->status, sizeof h, cudaMemcpyDeviceToHost, st), "status copy");
    if (s == TR_OK) s = cuda_check(cudaStreamSynchronize(st), "walk kernels");
    if (s != TR_OK) return s;
    if (h[2] > 0) return set_error(TR_EINVAL, "%d target index(es) outside [0, %lld)", h[2], (long long)t->n_cells);
    if (h[0] > 0)
        return set_error(TR_EOVERFLOW, "the walk stack overflowed for %d target(s); their outputs are NaN", h[0]);
    return TR_OK;
}

}  // namespace tr
