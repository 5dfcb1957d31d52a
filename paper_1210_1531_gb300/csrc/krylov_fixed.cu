// a3 + a4 in 57-bit fixed point on the integer pipe: the per-column Krylov build of krylov.cu,
// the same recursion (krylov.cu's header) on vectors held as integers with one power-of-two scale
// each, for Slater-Koster systems and for a caller's H and S.
//
// Why integers: the FP64 pipe of this chip retires 1.68 FMA per clock and SM, and the FP64 form of
// the recursion keeps it 92% busy, so no layout makes that form faster. The 32 x 32 + 64-bit integer
// multiply-add (mad.wide) retires 33 to 36 per clock and SM, and three of them make one product
// of two 57-bit numbers, so the same work costs a seventh of the pipe time.
//
// Numbers. A vector is x_i = f V_i with one double f and integers |V_i| <= 2^56 scaled so that the
// largest lies in (2^55, 2^56]; V = h 2^28 + l is stored as two 32-bit words (8 bytes, as a double).
// A product is V V' / 2^56 = h h' + (h l' + l h') / 2^28, the l l' term (below 2^-58 of the largest
// product) dropped; h h' and the cross terms are summed exactly in two 64-bit accumulators. So
// a dot product has no rounding but that of the dropped terms and one rounding per partial sum
// (2^-57 of the largest product; FP64 rounds every partial sum), and a vector is rounded to
// 2^-57 of its largest entry (FP64: each entry to 2^-53 of itself). Sums of integers
// do not depend on their order: a form's results are the same for every grid, queue and batch (the two
// forms, fx_form_for, cut their partial sums differently). Scalars
// (norms, H', S', Gram-Schmidt coefficients) are FP64, and so are the vectors of the first steps (the lead,
// at kLead).
//
// Coefficients of the two-centre blocks carry one power-of-two scale per matrix (FxScale): the
// largest is below 2^57 and the sum of any row's bounds below 2^62 (2^60 for rows of 33 to 64
// blocks, whose cross terms add up further), so no sum of a sparse product overflows. This form is
// used only where every row sum lies within 2^5 of the largest, so that a row's coefficients keep 52 bits
// of its largest at least (one of FP64's 53), and those of rows within 2^4 as many as FP64 gives. Here the
// row sums of H differ by up to 14 (graphite with grains), of S by up to 5. A caller's dense blocks
// are held alike, by exact row sums, up to 32 blocks a row: four products a row and block.
//
// The host reads whether the form suits a Slater-Koster system when it is built. elses_set_hs does not
// wait for the device, so with a caller's matrices both kernels are launched and the device decides:
// the one that is not to run returns at once.
//
// Against an 80-bit recursion (48 columns of 512-atom systems, G at three energies, geometric mean
// of the relative errors; FP64 kernel and the longer chase first): displaced diamond 7.7e-15 / 7.1e-15
// with two classical passes and 8.7e-15 / 8.0e-15 with the second from S'; dense disordered carbon 1.11e-14 /
// 1.18e-14 and 1.19e-14 / 1.17e-14; the same H and S as a caller's: 8.3e-15 / 7.2e-15, 7.9e-15 / 7.5e-15,
// 1.12e-14 / 1.10e-14, 1.04e-14 / 1.31e-14. rho of 256 columns of graphite with grains: geometric mean
// 7.0e-16 / 6.8e-16, largest 1.1e-14 / 3.7e-14 (one column). rho with one way of Gram-Schmidt against the other, all
// columns, root mean square: graphite with grains 1.6e-15 / 0.8e-15, diamond (4096) 5.1e-16 / 2.9e-16,
// disordered carbon (4096) 3.1e-15 / 4.7e-15; poles, median 4 to 11e-14 / 2 to 4e-14 eV.
#include <algorithm>

#include "krylov.cuh"
#include "krylov_fixed.cuh"

namespace elses {

// ------------------------------------------------------------------------------ coefficients
// Per atom: the bound on the absolute row sums of H and S in the two-centre form (every product
// of the block's arithmetic counted; |u . x| <= sqrt(3) max |x|), and the largest coefficients.
// out: [0] max row H, [1] max row S, [2] max |coefficient| H, [3] S, [4] complement of the
// smallest row H, [5] of the smallest row S, as bits of non-negative doubles (ordered like integers).
__global__ void k_fx_bounds(int n, const int* __restrict__ row_ptr, const int* __restrict__ col_idx,
                            const double* __restrict__ skr, double Es, double Ep, unsigned long long* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (i < n) {
        v[2] = fmax(fabs(Es), fabs(Ep));
        v[3] = 1.0;
        v[0] = v[2];
        v[1] = 1.0;
        bool finite = isfinite(Es) && isfinite(Ep);   // (fmax drops a NaN)
        for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            if (col_idx[e] == i) continue;
            const double* q = skr + 12 * (size_t)e;
            for (int m = 0; m < 2; ++m) {
                const double ss = fabs(q[4 + 4 * m]), sp = fabs(q[5 + 4 * m]);
                const double pi = fabs(q[6 + 4 * m]), dv = fabs(q[7 + 4 * m]);
                v[m] += fmax(ss, pi) + 1.75 * (sp + dv);
                v[2 + m] = fmax(v[2 + m], fmax(fmax(ss, sp), fmax(pi, dv)));
                finite = finite && ss + sp + pi + dv <= 1e300;
            }
            // u: the direction, not a number between atoms in one place
            const double* u = skr + 12 * (size_t)e;
            finite = finite && fabs(u[0]) + fabs(u[1]) + fabs(u[2]) <= 2.0;
        }
        // NaN and infinities are recorded as the largest value: the FP64 kernels then run and report them
        if (!finite) v[0] = v[1] = v[2] = v[3] = 1e308;
    }
    unsigned long long w[6];
    for (int m = 0; m < 4; ++m) w[m] = (unsigned long long)__double_as_longlong(v[m]);
    w[4] = i < n ? ~w[0] : 0ull;
    w[5] = i < n ? ~w[1] : 0ull;
    for (int m = 0; m < 6; ++m) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, w[m], o);
            w[m] = x > w[m] ? x : w[m];
        }
        if ((threadIdx.x & 31) == 0) atomicMax(out + m, w[m]);
    }
}

__device__ __forceinline__ long long fx_round(double v, int e) { return llrint(ldexp(v, e)); }

// The scales, and whether the fixed-point form is used (FxScale::ok, read by the host).
// dense: no product of the block is itself multiplied again, so coefficients may be twice as large;
// four products a row and block limit rows to 32 blocks.
__global__ void k_fx_scale(const unsigned long long* b, double Es, double Ep, int max_row, int dense, FxScale* out) {
    double v[4], lo[2];
    for (int m = 0; m < 4; ++m) v[m] = __longlong_as_double((long long)b[m]);
    for (int m = 0; m < 2; ++m) lo[m] = __longlong_as_double((long long)~b[4 + m]);
    FxScale s{};
    s.ok = max_row <= (dense ? 32 : 64);
    for (int m = 0; m < 2; ++m)
        if (!(v[m] > 1e-100 && v[m] < 1e100 && v[m] <= 32.0 * lo[m] && v[2 + m] > 0.0)) s.ok = 0;
    // the second Gram-Schmidt pass takes its coefficients, of order 2^63 sqrt(S), to single precision
    if (!(v[1] > 0x1p-60 && v[1] < 0x1p60)) s.ok = 0;
    if (s.ok) {
        const int row_bits = max_row <= 32 ? 61 : 59;
        s.eH = min(56 + dense - ilogb(v[2]), row_bits - ilogb(v[0]));
        s.eS = min(56 + dense - ilogb(v[3]), row_bits - ilogb(v[1]));
        s.Es = fx_split(fx_round(Es, s.eH));
        s.Ep = fx_split(fx_round(Ep, s.eH));
        s.one = fx_split(fx_round(1.0, s.eS));
    }
    *out = s;
}

// Block records for the sparse products, 96 bytes each: u (three words of scale 2^56, one unused),
// then (ss, sp, pp_pi, pp_sigma - pp_pi) of H and of S in their matrices' scales.
__global__ void k_fx_records(int nnzb, const double* __restrict__ skr, const FxScale* __restrict__ sc,
                             int2* __restrict__ rec) {
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= 12 * (size_t)nnzb || !sc->ok) return;
    const int m = (int)(q % 12);
    rec[q] = fx_split(fx_round(skr[q], m < 4 ? 56 : m < 8 ? sc->eH : sc->eS));
}

// The same of caller matrices, dense 4 x 4 blocks: exact absolute row sums.
__global__ void k_fx_bounds_dense(int n, const int* __restrict__ row_ptr, const double* __restrict__ H,
                                  const double* __restrict__ S, unsigned long long* out) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x, i = q >> 2, r = q & 3;
    unsigned long long w[6] = {0, 0, 0, 0, 0, 0};
    if (i < n) {
        for (int m = 0; m < 2; ++m) {
            const double* X = m ? S : H;
            double sum = 0.0, mx = 0.0;
            for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e)
                for (int c = 0; c < 4; ++c) {
                    const double v = fabs(X[16 * (size_t)e + 4 * r + c]);
                    sum += v;
                    mx = fmax(mx, v);
                }
            if (!(sum <= 1e300)) sum = mx = 1e308;
            w[m] = (unsigned long long)__double_as_longlong(sum);
            w[2 + m] = (unsigned long long)__double_as_longlong(mx);
            w[4 + m] = ~w[m];
        }
    }
    for (int m = 0; m < 6; ++m) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, w[m], o);
            w[m] = x > w[m] ? x : w[m];
        }
        if ((threadIdx.x & 31) == 0) atomicMax(out + m, w[m]);
    }
}

// Block records of caller matrices, 256 bytes each: H then S, row by row.
__global__ void k_fx_records_dense(int nnzb, const double* __restrict__ H, const double* __restrict__ S,
                                   const FxScale* __restrict__ sc, int2* __restrict__ rec) {
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= 32 * (size_t)nnzb || !sc->ok) return;
    const size_t e = q >> 5, m = q & 31;
    rec[q] = m < 16 ? fx_split(fx_round(H[16 * e + m], sc->eH)) : fx_split(fx_round(S[16 * e + m - 16], sc->eS));
}

void fx_build_dense(int n, int nnzb, const int* row_ptr, const double* H, const double* S, int max_row,
                    unsigned long long* bounds, FxScale* scale, int2* rec, cudaStream_t st) {
    cudaMemsetAsync(bounds, 0, 6 * sizeof(unsigned long long), st);
    k_fx_bounds_dense<<<(4 * n + 127) / 128, 128, 0, st>>>(n, row_ptr, H, S, bounds);
    k_fx_scale<<<1, 1, 0, st>>>(bounds, 0.0, 0.0, max_row, 1, scale);
    const size_t w = 32 * (size_t)nnzb;
    k_fx_records_dense<<<(unsigned)((w + 255) / 256), 256, 0, st>>>(nnzb, H, S, scale, rec);
}

void fx_build(int n, int nnzb, const int* row_ptr, const int* col_idx, const double* skr, double Es, double Ep,
              int max_row, unsigned long long* bounds, FxScale* scale, int2* rec, cudaStream_t st) {
    cudaMemsetAsync(bounds, 0, 6 * sizeof(unsigned long long), st);
    k_fx_bounds<<<(n + 127) / 128, 128, 0, st>>>(n, row_ptr, col_idx, skr, Es, Ep, bounds);
    k_fx_scale<<<1, 1, 0, st>>>(bounds, Es, Ep, max_row, 0, scale);
    const size_t w = 12 * (size_t)nnzb;
    k_fx_records<<<(unsigned)((w + 255) / 256), 256, 0, st>>>(nnzb, skr, scale, rec);
}

// ------------------------------------------------------------------------------ the kernel
// One CTA of T threads per atom, NC of its four columns at a time. Vectors of the NC columns are
// interleaved: unit (16 bytes) = two orbitals of one column; unit index = (2 a + half) NC + column,
// a the atom's place in the sorted cluster, half (orbitals 0, 1 or 2, 3) swapped on odd a / 2 so that
// the sparse products' gathers spread over the banks. Unit u belongs to thread u mod T in every
// dense sweep, so a basis vector is written and read by the same thread and sweeps need no
// barrier; the column of a thread is its index mod NC. In the sparse products a group of NC
// neighbouring threads owns rows (atoms), one column each, and the block records are read once
// for the NC columns.
//
// The basis U is read twice per step and SU once. Since the units are thread-private, the first
// vectors of U live in tensor memory (256 KB an SM, used as plain storage: a unit is four
// columns of the thread's lane), the next in the shared memory the work arrays leave, the rest
// and SU in per-CTA global scratch.
template <int NC>
__device__ __forceinline__ int fx_unit(int a, int half, int col) {
    return (2 * a + (half ^ ((a >> 1) & 1))) * NC + col;
}

// Offsets of the work arrays in dynamic shared memory.
struct FxLayout {
    unsigned X, P, Y;       // int4[units]: u_n, H u_n (then w) and S u_n
    unsigned g;             // int2[NC][nu]: update coefficients
    unsigned f, s, h, E;    // double[NC][nu]: scales of U and of SU (times 2^60), coefficients; [NC][packed]: S' - I
    unsigned hf, Ef;        // float: h and E in single precision
    unsigned row;           // int2[3][NC][nu]: entry j of the integer vectors X, Y, P of every step
    unsigned ex;            // int[2][NC][nu]: exponents, S u_n = f 2^ex Y and H u_n = f 2^ex P
    unsigned red;           // int[3][NC][3 nu + 1]: sums of the dot products in three pieces
    unsigned cl, base, off, deg;   // int[na (+ 1)]: atoms, first block, first entry, entries of each row
    unsigned ent;           // entries: byte offsets of the neighbour's first unit (<< 16) and of the
                            // block's record within its row
    unsigned row_at;        // short[slots][groups]: rows of each group
    unsigned at;            // short: places in the cluster of the pattern row of J
    unsigned pos, pos_atom; // int: the exact gradient's positions of the cluster's atoms, and back (kept bases only)
    unsigned cache;         // int4: basis vectors
};

template <int NC, int T>
__host__ __device__ inline FxLayout fx_layout(int na, int nu, int max_row, bool overlap, bool store) {
    FxLayout v;
    unsigned o = 0;
    const int G = T / NC, ns = (na + G - 1) / G, pk = overlap ? nu * (nu + 1) / 2 : 0;
    auto take = [&](size_t bytes) { const unsigned at = o; o += (unsigned)((bytes + 15) & ~(size_t)15); return at; };
    v.X = take(sizeof(int4) * 2 * NC * na);
    v.P = take(sizeof(int4) * 2 * NC * na);
    v.Y = take(sizeof(int4) * 2 * NC * na);
    v.g = take(sizeof(int2) * NC * nu);
    v.f = take(sizeof(double) * NC * nu);
    v.s = take(sizeof(double) * NC * nu);
    v.h = take(sizeof(double) * NC * nu);
    v.E = take(sizeof(double) * NC * pk);
    v.hf = take(sizeof(float) * NC * nu);
    v.Ef = take(sizeof(float) * NC * pk);
    v.row = take(sizeof(int2) * 3 * NC * nu);
    v.ex = take(sizeof(int) * 2 * NC * nu);
    v.red = take(sizeof(int) * 3 * NC * (3 * nu + 1));
    v.cl = take(sizeof(int) * na);
    v.base = take(sizeof(int) * na);
    v.off = take(sizeof(int) * (na + 1));
    v.deg = take(sizeof(int) * na);
    v.ent = take(sizeof(unsigned) * (size_t)na * max_row);
    v.row_at = take(sizeof(short) * ns * G);
    v.at = take(sizeof(short) * max_row);
    v.pos = take(store ? sizeof(int) * na : 0);
    v.pos_atom = take(store ? sizeof(int) * (na + 32) : 0);
    v.cache = o;
    return v;
}

extern __shared__ __align__(16) unsigned char fx_smem[];
template <class E>
__device__ __forceinline__ E* fx_at(unsigned off) {
    return reinterpret_cast<E*>(fx_smem + off);
}

// What the phases of a step share, in shared memory: the phases are functions of their own, each with
// the registers to itself.
template <int NC>
struct FxState {
    FxLayout v;
    FxScale sc;
    const int4* rec;
    int4 *gU, *gY;          // basis vectors in global scratch, `units` apart
    double2 *gD, *hd;       // lead: the vectors in FP64 (in units of X), `units` apart, and H u_n, then w
    double2* xa;            // shared memory for the first kLead + 1 of them in turn, or null
    unsigned tmem;
    int n_at, NS, units, upt, qJ, nent, nu, nm, alpha0;
    int kT, kS, kY;         // U[0, kT) in tensor memory, U[kT, kS) and SU[0, kY) in shared memory
    bool overlap;
    int atom, live;
    int slot;               // of the atom's columns in the store of bases
    unsigned long long bits[2][NC];   // or of the magnitudes of new vectors
    unsigned top[2][NC];    // the same of the lead's FP64 vectors: largest high word
    int bH[NC], bS[NC];     // H u_n = f 2^bH P, S u_n = f 2^bS Y
    int sP[NC];             // lead: P = xd 2^sP, rounded
    int lead, small;        // steps of the lead; whether an atom is still too small to leave it
    double Es, Ep;
    double hh[2][NC];       // |P|^2 of the even and the odd steps
    int q[NC], done[NC], nue[NC], we[NC], big[NC];
};

// Shift that brings values whose absolute values or to m below 2^56, the largest above 2^55.
__device__ __forceinline__ int fx_shift(unsigned long long m) { return m ? 8 - __clzll((long long)m) : 0; }
__device__ __forceinline__ long long fx_norm(long long v, int sh) {
    return sh > 0 ? (v + (1ll << (sh - 1))) >> sh : v << -sh;
}
__device__ __forceinline__ int4 fx_norm2(longlong2 v, int sh) {
    const int2 a = fx_split(fx_norm(v.x, sh)), b = fx_split(fx_norm(v.y, sh));
    return make_int4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ unsigned long long fx_abs_bits(long long v) { return (unsigned long long)(v ^ (v >> 63)); }
// 2^e as a double without FP64 instructions (e within the normal range)
__device__ __forceinline__ double fx_pow2(int e) {
    return __longlong_as_double((long long)(1023 + max(-1022, min(1023, e))) << 52);
}

// or of m over the lanes of a warp that hold the same column, then into the column's word
template <int NC>
__device__ __forceinline__ void fx_or(unsigned long long m, unsigned long long* to) {
    unsigned hi = (unsigned)(m >> 32), lo = (unsigned)m;
#pragma unroll
    for (int o = NC; o < 32; o <<= 1) {
        hi |= __shfl_xor_sync(0xffffffffu, hi, o);
        lo |= __shfl_xor_sync(0xffffffffu, lo, o);
    }
    if ((threadIdx.x & 31) < NC) {
        unsigned* w = reinterpret_cast<unsigned*>(to);
        atomicOr(w, lo);
        atomicOr(w + 1, hi);
    }
}

// The largest m over the lanes of a warp that hold the same column, then into the column's word
template <int NC>
__device__ __forceinline__ void fx_max(unsigned m, unsigned* to) {
#pragma unroll
    for (int o = NC; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) < NC) atomicMax(to, m);
}
__device__ __forceinline__ bool fx_zero(const double2 v) { return v.x == 0.0 && v.y == 0.0; }
__device__ __forceinline__ unsigned fx_top(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
// s with 2^55 <= 2^s v < 2^56 for the largest v, of high word `top`
__device__ __forceinline__ int fx_lead_shift(unsigned top) { return top ? 55 - ((int)(top >> 20) - 1023) : 0; }
__device__ __forceinline__ int4 fx_lead_split(const double2 v, double scale) {
    const int2 a = fx_split(__double2ll_rn(v.x * scale)), b = fx_split(__double2ll_rn(v.y * scale));
    return make_int4(a.x, a.y, b.x, b.y);
}

// Sums of the 8 values of every lane over eight lanes of the warp with the same column, by recursive
// halving (eight, so that the sum of units of up to 2^56 fits 64 bits): every lane ends with the sum
// of one value, whose index it returns, in v[0]; NC = 2 in two parts per value (one per
// half-warp), NC = 1 in four.
template <int NC>
__device__ __forceinline__ int fx_sum(long long (&v)[8]) {
    const int lane = threadIdx.x & 31;
    int first = 0, o = 4 * NC;
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
        if (up) first += w;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const long long send = up ? v[i] : v[i + w], keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return first;
}

// A 64-bit sum into three 32-bit shared words (22, 21 and 21 bits), and back as a double.
__device__ __forceinline__ void fx_red_add(int* r, int stride, long long v) {
    atomicAdd(r, (int)(v >> 42));
    atomicAdd(r + stride, (int)(v >> 21) & 0x1fffff);
    atomicAdd(r + 2 * stride, (int)v & 0x1fffff);
}
__device__ __forceinline__ double fx_red_get(const int* r, int stride) {
    const long long top = r[0], mid = r[stride], lo = r[2 * stride];
    // sums over the warps of up to 63 bits are exact; longer ones (of vectors whose entries nearly
    // all have the largest magnitude) drop four low bits
    const bool fits = (unsigned)(r[0] + (1 << 20)) < (2u << 20);
    const long long q = fits ? (top << 42) + (mid << 21) + lo : (top << 38) + (((mid << 21) + lo + 8) >> 4);
    const double v = (double)q;
    return fits && q != 0 ? __hiloint2double(__double2hiint(v) - (4 << 20), __double2loint(v)) : v;   // times 2^-4
}

__device__ __forceinline__ int2 fx_lo(const int4& v) { return make_int2(v.x, v.y); }
__device__ __forceinline__ int2 fx_hi(const int4& v) { return make_int2(v.z, v.w); }

// The lead: first steps whose vectors are formed and kept in FP64 beside the integers, which then serve the
// dot products only. A step reaches the next shell of the cluster with amplitudes far below the vector's
// largest (2^-18 two bonds on; 2^-20 to 2^-70 behind a bond near the cutoff), which FP64 holds to 53
// bits of themselves and the integers only to 2^-57 of the largest; where the cluster has a state
// there, the later steps amplify what was lost. So the lead lasts kLead steps, and on while one of the CTA's
// columns still reaches new atoms or has an atom below 2^-kSmall of the largest in its last two vectors.
// Largest pole errors against an 80-bit recursion, in eV, of the 28 to 70 columns where the kernels
// differ most, FP64 kernel first: graphite with diamond grains (32768 atoms) 2.6e-10 / 2.6e-10, dense
// disordered carbon (4096) 1.2e-10 / 1.0e-10, diamond (4096) 5.6e-11 / 5.7e-11. (With six steps whatever
// the amplitudes, and their vectors subtracted as integers, the first was 1.2e-9 and rho there off by 6e-12.)
// Each step costs 3% of the kernel. kLead 6 and kSmall 10, in ms: diamond 33.3 (32.9 with six steps
// always), disordered carbon (65536) 303 (299), graphite with grains 184 (154): a third of its atoms have
// neighbours behind weak bonds. kSmall 12: 177 there, but poles off by 3.0e-10; kSmall 8: 193, 34.3 and 314.
constexpr int kLead = 6, kSmall = 10;

template <int T, int kMinB>
struct FxTmem {
    // whole groups of four warps share the columns, and an allocation is a power of two
    static_assert(T % 128 == 0 && (kMinB == 1 || kMinB == 2), "tensor memory split");
    static constexpr int cols = 512 / kMinB;                              // of a CTA
    static constexpr int units = cols / (T / 128) / 4;                     // a thread can keep there
    __device__ static unsigned base(unsigned at) {
        const int warp = threadIdx.x >> 5;
        return at + ((unsigned)(warp & 3) << 21) + (warp >> 2) * (4 * units);
    }
};

// The cluster of atom J: atoms, entries, and the rows of each group. Every thread of the CTA calls it.
template <int NC, int T, bool kDense>
__device__ __forceinline__ void fx_view(const KrylovArgs& a, FxState<NC>& st, int J, int cbase, int n_at) {
    constexpr int G = T / NC;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int *cl = fx_at<int>(st.v.cl), *base = fx_at<int>(st.v.base), *off = fx_at<int>(st.v.off), *deg = fx_at<int>(st.v.deg);
    unsigned* ent = fx_at<unsigned>(st.v.ent);
    short *row_at = fx_at<short>(st.v.row_at), *at = fx_at<short>(st.v.at);
    for (int q = tid; q < n_at; q += T) {
        const int A = a.cl_ptr ? a.cl_idx[cbase + q] : q;
        cl[q] = A;
        base[q] = a.row_ptr[A];
        deg[q] = a.row_ptr[A + 1] - a.row_ptr[A];
        if (A == J) st.qJ = q;
    }
    __syncthreads();
    if (warp == 0) {                              // places of the rows' entries
        int sum = 0;
        for (int q0 = 0; q0 < n_at; q0 += 32) {
            int d = q0 + lane < n_at ? deg[q0 + lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, d, o);
                if (lane >= o) d += t;
            }
            if (q0 + lane < n_at) off[q0 + lane + 1] = sum + d;
            sum += __shfl_sync(0xffffffffu, d, 31);
        }
        if (lane == 0) off[0] = 0;
    }
    __syncthreads();
    const int qJ = st.qJ;
    // in-cluster off-site entries of each row: a warp takes four rows at a time so that their
    // loads and searches overlap
    int top = 1;                                  // largest power of two <= n_at
    while (2 * top <= n_at) top *= 2;
    for (int q0 = 4 * warp; q0 < n_at; q0 += 4 * (T / 32)) {
        int cnt[4] = {0, 0, 0, 0}, len = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (q0 + i < n_at) len = max(len, off[q0 + i + 1] - off[q0 + i]);
        for (int r0 = 0; r0 < len; r0 += 32) {
            const int r = r0 + lane;
            int ce[4], pos[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool in = q0 + i < n_at && r < off[q0 + i + 1] - off[q0 + i];
                ce[i] = in ? a.col_idx[base[q0 + i] + r] : -1;
                pos[i] = -1;                      // last place with cl <= ce
            }
            for (int sp = top; sp > 0; sp >>= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (pos[i] + sp < n_at && cl[pos[i] + sp] <= ce[i]) pos[i] += sp;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int q = q0 + i;
                if (q >= n_at) break;
                const bool in = ce[i] >= 0 && pos[i] >= 0 && cl[pos[i]] == ce[i];
                if (q == qJ && in) at[r] = (short)pos[i];
                const unsigned hit = __ballot_sync(0xffffffffu, in && (kDense || pos[i] != q));
                if (in && (kDense || pos[i] != q))
                    ent[off[q] + cnt[i] + __popc(hit & ((1u << lane) - 1u))] =
                        ((unsigned)fx_unit<NC>(pos[i], 0, 0) << 20) | (unsigned)(r * (kDense ? 256 : 96));
                cnt[i] += __popc(hit);
            }
        }
        __syncwarp();
        if (lane < 4 && q0 + lane < n_at) deg[q0 + lane] = lane == 0 ? cnt[0] : lane == 1 ? cnt[1] : lane == 2 ? cnt[2] : cnt[3];
    }
    const int NS = (n_at + G - 1) / G;
    for (int q = tid; q < NS * G; q += T) row_at[q] = -1;
    __syncthreads();
    // rows in decreasing degree, dealt to the groups there and back again: the threads of a
    // warp walk rows of nearly equal length, and the groups' totals balance
    int nent_part = 0;
    for (int q = tid; q < n_at; q += T) {
        const int dq = deg[q];
        int rank = 0;
        for (int b = 0; b < n_at; ++b) {
            const int db = deg[b];
            rank += (db > dq) || (db == dq && b < q);
        }
        const int sl = rank / G, g = rank % G;
        row_at[sl * G + ((sl & 1) ? G - 1 - g : g)] = (short)q;
        nent_part += dq;
    }
    if (nent_part) atomicAdd(&st.nent, nent_part);
    __syncthreads();
    if (tid == 0) st.NS = NS;
}

// H X and S X: each thread forms its column's entries of its group's rows, as 64-bit sums into P and Y.
template <int NC, int T>
__device__ __forceinline__ void fx_products(FxState<NC>& st) {
    constexpr int G = T / NC;
    const int tid = threadIdx.x, tc = tid % NC, NS = st.NS;
    const int4* X = fx_at<int4>(st.v.X);
    const short* row_at = fx_at<short>(st.v.row_at);
    unsigned long long mH = 0, mS = 0;
    const int g = tid / NC;
    longlong2* PH = fx_at<longlong2>(st.v.P);
    longlong2* PS = fx_at<longlong2>(st.v.Y);
    const char* const Xc = reinterpret_cast<const char*>(X + tc);
#pragma unroll 1
    for (int sl = 0; sl < NS; ++sl) {
        const int q = row_at[sl * G + g];
        if (q < 0) continue;
        const unsigned* ent = fx_at<unsigned>(st.v.ent) + fx_at<int>(st.v.off)[q];
        const char* rb = reinterpret_cast<const char*>(st.rec + 6 * (size_t)fx_at<int>(st.v.base)[q]);
        const int d = fx_at<int>(st.v.deg)[q];
        // two entries' records are in flight: one being applied, the next being fetched
        int4 ra[6], rc[6];
        unsigned ea = 0, ec = 0;
        auto fetch = [&](int k, unsigned& en, int4 (&r)[6]) {
            en = d > 0 ? ent[min(k, d - 1)] : 0u;     // past the end: the last entry's record again
            const int4* at = reinterpret_cast<const int4*>(rb + (en & 0xffffu));
#pragma unroll
            for (int i = 0; i < 6; ++i) r[i] = __ldg(at + i);
        };
        fetch(0, ea, ra);
        const int u01 = fx_unit<NC>(q, 0, tc), u23 = fx_unit<NC>(q, 1, tc);
        Fx H0, H1, H2, H3, S0, S1, S2, S3;
        {
            const int4 a01 = X[u01], a23 = X[u23];
            fx_mul(H0, st.sc.Es, fx_lo(a01));
            fx_mul(H1, st.sc.Ep, fx_hi(a01));
            fx_mul(H2, st.sc.Ep, fx_lo(a23));
            fx_mul(H3, st.sc.Ep, fx_hi(a23));
            fx_mul(S0, st.sc.one, fx_lo(a01));
            fx_mul(S1, st.sc.one, fx_hi(a01));
            fx_mul(S2, st.sc.one, fx_lo(a23));
            fx_mul(S3, st.sc.one, fx_hi(a23));
        }
        auto apply = [&](unsigned en, const int4 (&c)[6]) {
            const unsigned at = en >> 16;
            const int4 b01 = *reinterpret_cast<const int4*>(Xc + at);
            const int4 b23 = *reinterpret_cast<const int4*>(Xc + (at ^ (16u * NC)));
            const int2 x0 = fx_lo(b01), x1 = fx_hi(b01), x2 = fx_lo(b23), x3 = fx_hi(b23);
            const int2 nx0 = make_int2(-x0.x, -x0.y);
            const int2 u0 = fx_lo(c[0]), u1 = fx_hi(c[0]), u2 = fx_lo(c[1]);
            // t = u . x_p; y_s += V_ss x_s + V_sp t; y_p += V_pi x_p + (dV t - V_sp x_s) u
            Fx tt, aa, ab;
            fx_mul_half(tt, u0, x1);
            fx_mac(tt, u1, x2);
            fx_mac(tt, u2, x3);
            fx_mul_half(aa, fx_hi(c[2]), nx0);
            fx_mul_half(ab, fx_hi(c[4]), nx0);
            const int2 t = fx_pair(tt);
            fx_mac(aa, fx_hi(c[3]), t);
            fx_mac(ab, fx_hi(c[5]), t);
            fx_mac(H0, fx_lo(c[2]), x0);
            fx_mac(S0, fx_lo(c[4]), x0);
            fx_mac(H1, fx_lo(c[3]), x1);
            fx_mac(S1, fx_lo(c[5]), x1);
            fx_mac(H2, fx_lo(c[3]), x2);
            fx_mac(S2, fx_lo(c[5]), x2);
            fx_mac(H3, fx_lo(c[3]), x3);
            fx_mac(S3, fx_lo(c[5]), x3);
            const int2 wh = fx_pair(aa), ws = fx_pair(ab);
            fx_mac(H0, fx_hi(c[2]), t);
            fx_mac(S0, fx_hi(c[4]), t);
            fx_mac(H1, wh, u0);
            fx_mac(S1, ws, u0);
            fx_mac(H2, wh, u1);
            fx_mac(S2, ws, u1);
            fx_mac(H3, wh, u2);
            fx_mac(S3, ws, u2);
        };
#pragma unroll 1
        for (int k = 0; k < d; k += 2) {
            fetch(k + 1, ec, rc);
            apply(ea, ra);
            if (k + 1 >= d) break;
            fetch(k + 2, ea, ra);
            apply(ec, rc);
        }
        longlong2 y01 = make_longlong2(fx_fold(H0), fx_fold(H1)), y23 = make_longlong2(fx_fold(H2), fx_fold(H3));
        mH |= fx_abs_bits(y01.x) | fx_abs_bits(y01.y) | fx_abs_bits(y23.x) | fx_abs_bits(y23.y);
        PH[u01] = y01;
        PH[u23] = y23;
        y01 = make_longlong2(fx_fold(S0), fx_fold(S1));
        y23 = make_longlong2(fx_fold(S2), fx_fold(S3));
        mS |= fx_abs_bits(y01.x) | fx_abs_bits(y01.y) | fx_abs_bits(y23.x) | fx_abs_bits(y23.y);
        PS[u01] = y01;
        PS[u23] = y23;
    }
    __syncwarp();
    fx_or<NC>(mH, &st.bits[0][tc]);
    fx_or<NC>(mS, &st.bits[1][tc]);
}

// The same with dense 4 x 4 blocks, the on-site ones among the entries: 32 products an entry instead of
// 16, 256 bytes of it instead of 96, which L2 has to deliver. H's block is applied while S's is on its
// way, and S's while the next entry's H is. 512 atoms, nu 30, set_hs to density matrix: 27.9 ms with the
// FP64 kernel, 11.9 ms (Slater-Koster form: 11.0 ms).
template <int NC, int T>
__device__ __forceinline__ void fx_products_dense(FxState<NC>& st) {
    constexpr int G = T / NC;
    const int tid = threadIdx.x, tc = tid % NC, g = tid / NC, NS = st.NS;
    const short* row_at = fx_at<short>(st.v.row_at);
    const char* const Xc = reinterpret_cast<const char*>(fx_at<int4>(st.v.X) + tc);
    longlong2 *PH = fx_at<longlong2>(st.v.P), *PS = fx_at<longlong2>(st.v.Y);
    unsigned long long mH = 0, mS = 0;
#pragma unroll 1
    for (int sl = 0; sl < NS; ++sl) {
        const int q = row_at[sl * G + g];
        if (q < 0) continue;
        const unsigned* ent = fx_at<unsigned>(st.v.ent) + fx_at<int>(st.v.off)[q];
        const char* rb = reinterpret_cast<const char*>(st.rec + 16 * (size_t)fx_at<int>(st.v.base)[q]);
        const int d = fx_at<int>(st.v.deg)[q], u01 = fx_unit<NC>(q, 0, tc), u23 = fx_unit<NC>(q, 1, tc);
        Fx H[4], S[4];
        int4 hb[8], sb[8];
        auto fetch = [&](unsigned en, int half, int4 (&b)[8]) {
            const int4* at = reinterpret_cast<const int4*>(rb + (en & 0xffffu)) + 8 * half;
#pragma unroll
            for (int i = 0; i < 8; ++i) b[i] = __ldg(at + i);
        };
        auto apply = [&](Fx (&y)[4], const int4 (&b)[8], const int4& x01, const int4& x23) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                fx_mac(y[r], fx_lo(b[2 * r]), fx_lo(x01));
                fx_mac(y[r], fx_hi(b[2 * r]), fx_hi(x01));
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                fx_mac(y[r], fx_lo(b[2 * r + 1]), fx_lo(x23));
                fx_mac(y[r], fx_hi(b[2 * r + 1]), fx_hi(x23));
            }
        };
        unsigned en = d > 0 ? ent[0] : 0u;
        if (d > 0) fetch(en, 0, hb);
#pragma unroll 1
        for (int k = 0; k < d; ++k) {
            fetch(en, 1, sb);
            const unsigned at = en >> 16;
            const int4 x01 = *reinterpret_cast<const int4*>(Xc + at);
            const int4 x23 = *reinterpret_cast<const int4*>(Xc + (at ^ (16u * NC)));
            apply(H, hb, x01, x23);
            en = ent[min(k + 1, d - 1)];
            fetch(en, 0, hb);
            apply(S, sb, x01, x23);
        }
        longlong2 y01 = make_longlong2(fx_fold(H[0]), fx_fold(H[1])), y23 = make_longlong2(fx_fold(H[2]), fx_fold(H[3]));
        mH |= fx_abs_bits(y01.x) | fx_abs_bits(y01.y) | fx_abs_bits(y23.x) | fx_abs_bits(y23.y);
        PH[u01] = y01;
        PH[u23] = y23;
        y01 = make_longlong2(fx_fold(S[0]), fx_fold(S[1]));
        y23 = make_longlong2(fx_fold(S[2]), fx_fold(S[3]));
        mS |= fx_abs_bits(y01.x) | fx_abs_bits(y01.y) | fx_abs_bits(y23.x) | fx_abs_bits(y23.y);
        PS[u01] = y01;
        PS[u23] = y23;
    }
    __syncwarp();
    fx_or<NC>(mH, &st.bits[0][tc]);
    fx_or<NC>(mS, &st.bits[1][tc]);
}

// The lead's form of fx_products: FP64 products of u_n into P and Y (as FP64), entries whose neighbour
// is not reached yet left out. An atom that is reached now keeps the lead going: there may be more behind it.
template <int NC, int T, bool kDense>
__device__ __forceinline__ void fx_products_lead(const KrylovArgs& a, FxState<NC>& st, int n) {
    constexpr int G = T / NC;
    const int tid = threadIdx.x, tc = tid % NC, g = tid / NC, NS = st.NS;
    const short* row_at = fx_at<short>(st.v.row_at);
    const double2* xd = n <= kLead && st.xa ? st.xa : st.gD + (size_t)n * st.units;
    const char* xc = reinterpret_cast<const char*>(xd + tc);
    double2 *PH = fx_at<double2>(st.v.P), *PS = fx_at<double2>(st.v.Y);
    unsigned mH = 0, mS = 0;
#pragma unroll 1
    for (int sl = 0; sl < NS; ++sl) {
        const int q = row_at[sl * G + g];
        if (q < 0) continue;
        const unsigned* ent = fx_at<unsigned>(st.v.ent) + fx_at<int>(st.v.off)[q];
        const size_t b0 = (size_t)fx_at<int>(st.v.base)[q];
        const char* rb = reinterpret_cast<const char*>(a.skr + 12 * b0);
        const int d = fx_at<int>(st.v.deg)[q], u01 = fx_unit<NC>(q, 0, tc), u23 = fx_unit<NC>(q, 1, tc);
        const double2 x01 = xd[u01], x23 = xd[u23];
        double2 s01 = make_double2(0.0, 0.0), s23 = s01;
        if (!kDense) {
            s01 = x01;
            s23 = x23;
        }
        double2 h01 = make_double2(st.Es * s01.x, st.Ep * s01.y), h23 = make_double2(st.Ep * s23.x, st.Ep * s23.y);
#pragma unroll 1
        for (int k = 0; k < d; ++k) {
            const unsigned en = ent[k], at = en >> 16;
            const double2 x01 = *reinterpret_cast<const double2*>(xc + at);
            const double2 x23 = *reinterpret_cast<const double2*>(xc + (at ^ (16u * NC)));
            if (fx_zero(x01) && fx_zero(x23)) continue;
            if (kDense) {
                const size_t e = 16 * (b0 + (en & 0xffffu) / 256);
                auto row = [&](const double* X, int r, double y) {
                    const double2 c01 = __ldg(reinterpret_cast<const double2*>(X + e + 4 * r));
                    const double2 c23 = __ldg(reinterpret_cast<const double2*>(X + e + 4 * r + 2));
                    return fma(c23.y, x23.y, fma(c23.x, x23.x, fma(c01.y, x01.y, fma(c01.x, x01.x, y))));
                };
                h01 = make_double2(row(a.H, 0, h01.x), row(a.H, 1, h01.y));
                h23 = make_double2(row(a.H, 2, h23.x), row(a.H, 3, h23.y));
                s01 = make_double2(row(a.S, 0, s01.x), row(a.S, 1, s01.y));
                s23 = make_double2(row(a.S, 2, s23.x), row(a.S, 3, s23.y));
                continue;
            }
            const double2* r = reinterpret_cast<const double2*>(rb + (en & 0xffffu));
            const double2 u = __ldg(r), uz = __ldg(r + 1), a01 = __ldg(r + 2), a23 = __ldg(r + 3);
            const double2 b01 = __ldg(r + 4), b23 = __ldg(r + 5);
            const double t = fma(uz.x, x23.y, fma(u.y, x23.x, u.x * x01.y));
            const double ah = fma(a23.y, t, -a01.y * x01.x), as = fma(b23.y, t, -b01.y * x01.x);
            h01.x = fma(a01.y, t, fma(a01.x, x01.x, h01.x));
            h01.y = fma(ah, u.x, fma(a23.x, x01.y, h01.y));
            h23.x = fma(ah, u.y, fma(a23.x, x23.x, h23.x));
            h23.y = fma(ah, uz.x, fma(a23.x, x23.y, h23.y));
            s01.x = fma(b01.y, t, fma(b01.x, x01.x, s01.x));
            s01.y = fma(as, u.x, fma(b23.x, x01.y, s01.y));
            s23.x = fma(as, u.y, fma(b23.x, x23.x, s23.x));
            s23.y = fma(as, uz.x, fma(b23.x, x23.y, s23.y));
        }
        if (n + 1 >= kLead && fx_zero(x01) && fx_zero(x23) && !(fx_zero(h01) && fx_zero(h23))) st.small = 1;
        mH = max(max(mH, max(fx_top(h01.x), fx_top(h01.y))), max(fx_top(h23.x), fx_top(h23.y)));
        mS = max(max(mS, max(fx_top(s01.x), fx_top(s01.y))), max(fx_top(s23.x), fx_top(s23.y)));
        PH[u01] = h01;
        PH[u23] = h23;
        PS[u01] = s01;
        PS[u23] = s23;
    }
    __syncwarp();
    fx_max<NC>(mH, &st.top[0][tc]);
    fx_max<NC>(mS, &st.top[1][tc]);
}

// Pass A of step n, X_k . HX_n and X_k . SX_n of the c <= 4 vectors from k0 (and |HX_n|^2 with the
// first) into the sums. x0: the vectors' first units, `units` apart (null: tensor memory). From
// memory, the next unit's vectors are fetched while one is applied. kFull: c = 4.
template <int NC, int T, int kMinB, bool kFull>
__device__ __forceinline__ void fx_dots_x(FxState<NC>& st, int k0, int c, const int4* x0) {
    const int tid = threadIdx.x, units = st.units, upt = st.upt;
    const int4 *P = fx_at<int4>(st.v.P) + tid, *Y = fx_at<int4>(st.v.Y) + tid;
    Fx acc[8], hh;
    auto apply = [&](int i, const int4 (&xv)[4]) {
        int4 p = make_int4(0, 0, 0, 0), y = p;
        if (tid + i * T < units) {
            p = P[i * T];
            y = Y[i * T];
        }
        if (k0 == 0) {
            fx_mac(hh, fx_lo(p), fx_lo(p));
            fx_mac(hh, fx_hi(p), fx_hi(p));
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
            if (kFull || kk < c) {
                fx_mac(acc[kk], fx_lo(xv[kk]), fx_lo(p));
                fx_mac(acc[4 + kk], fx_lo(xv[kk]), fx_lo(y));
                fx_mac(acc[kk], fx_hi(xv[kk]), fx_hi(p));
                fx_mac(acc[4 + kk], fx_hi(xv[kk]), fx_hi(y));
            }
    };
    if (!x0) {
        const unsigned tm = FxTmem<T, kMinB>::base(st.tmem) + 4 * k0 * upt;
#pragma unroll 1
        for (int i = 0; i < upt; ++i) {
            int4 xv[4];
            fx_tmem_ld<4>(tm + 4 * i, 4 * upt, xv);
            apply(i, xv);
        }
    } else {
        int4 xa[4], xb[4];
        auto load = [&](int i, int4 (&xv)[4]) {
            const int4* q = x0 + min(tid + i * T, units - 1);   // a unit past the end meets P = Y = 0
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                xv[kk] = *q;
                if (kFull || kk + 1 < c) q += units;
            }
        };
        load(0, xa);
#pragma unroll 1
        for (int i = 0; i < upt; i += 2) {
            load(i + 1, xb);
            apply(i, xa);
            load(i + 2, xa);
            apply(i + 1, xb);
        }
    }
    __syncwarp();
    long long s[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = fx_fold(acc[i]);
    const int val = fx_sum<NC>(s), k = val & 3, nm = st.nm, RC = 3 * nm + 1;
    int* red = fx_at<int>(st.v.red) + (tid % NC) * RC;
    if (k < c) fx_red_add(red + (val >> 2) * nm + k0 + k, NC * RC, s[0]);
    if (k0 == 0) {
        __syncwarp();
        long long h = fx_fold(hh);
#pragma unroll
        for (int o = NC; o < 8 * NC; o <<= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
        if (val == 0) fx_red_add(red + 3 * nm, NC * RC, h);
    }
    __syncwarp();
}

// The same of SX_k . w for the c <= 8 vectors from k0, w in P; y0: their first units. Sums of kind
// `kind` (2 in pass A, 0 in the second classical pass). kFull: c = 8.
template <int NC, int T, bool kFull>
__device__ __forceinline__ void fx_dots_y(FxState<NC>& st, int k0, int c, const int4* y0, int kind) {
    const int tid = threadIdx.x, units = st.units, upt = st.upt;
    const int4* P = fx_at<int4>(st.v.P) + tid;
    Fx acc[8];
    int4 ya[8], yb[8];
    auto load = [&](int i, int4 (&yv)[8]) {
        const int4* q = y0 + min(tid + i * T, units - 1);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            yv[kk] = *q;
            if (kFull || kk + 1 < c) q += units;
        }
    };
    auto apply = [&](int i, const int4 (&yv)[8]) {
        int4 p = make_int4(0, 0, 0, 0);
        if (tid + i * T < units) p = P[i * T];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
            if (kFull || kk < c) {
                fx_mac(acc[kk], fx_lo(yv[kk]), fx_lo(p));
                fx_mac(acc[kk], fx_hi(yv[kk]), fx_hi(p));
            }
    };
    load(0, ya);
#pragma unroll 1
    for (int i = 0; i < upt; i += 2) {
        load(i + 1, yb);
        apply(i, ya);
        load(i + 2, ya);
        apply(i + 1, yb);
    }
    __syncwarp();
    long long s[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = fx_fold(acc[i]);
    const int val = fx_sum<NC>(s), nm = st.nm, RC = 3 * nm + 1;
    if (val < c) fx_red_add(fx_at<int>(st.v.red) + (tid % NC) * RC + kind * nm + k0 + val, NC * RC, s[0]);
    __syncwarp();
}

// SX_k . w for k <= n, in runs that do not cross from shared memory to scratch.
template <int NC, int T>
__device__ __forceinline__ void fx_sweep_y(FxState<NC>& st, int n, int kind) {
    const int units = st.units;
#pragma unroll 1
    for (int k = 0; k <= n;) {
        const bool near = k < st.kY;
        const int end = min(min(k + 8, n + 1), near ? st.kY : n + 1);
        const int4* y0 = near ? fx_at<int4>(st.v.cache) + (st.kS - st.kT + k) * units : st.gY + (size_t)k * units;
        if (end - k == 8) fx_dots_y<NC, T, true>(st, k, 8, y0, kind);
        else fx_dots_y<NC, T, false>(st, k, end - k, y0, kind);
        k = end;
    }
}

template <int NC, int T, int kMinB>
__device__ __forceinline__ void fx_pass_a(FxState<NC>& st, int n) {
    const int units = st.units;
#pragma unroll 1
    for (int k = 0; k <= n;) {
        int end = min(k + 4, n + 1);
        const int4* x0 = nullptr;
        if (k < st.kT) {
            end = min(end, st.kT);
        } else if (k < st.kS) {
            end = min(end, st.kS);
            x0 = fx_at<int4>(st.v.cache) + (k - st.kT) * units;
        } else {
            x0 = st.gU + (size_t)k * units;
        }
        if (end - k == 4) fx_dots_x<NC, T, kMinB, true>(st, k, 4, x0);
        else fx_dots_x<NC, T, kMinB, false>(st, k, end - k, x0);
        k = end;
    }
    fx_sweep_y<NC, T>(st, n, 2);
}

// The scalars of column c after pass A of step n, by two warps. Dot products come in units of 2^60 of
// the integers' products; u_n = f X, S u_n = f 2^bS Y, H u_n = f 2^bH P.
//
// X^T S X, and whether u_n exists: the tests on w = 2^we X times the scale of H u_(n-1) (n > 0)
// against its norm, w^T S w against that of H u_(n-1), both without the common scale. Returns 0, 1
// (no new direction), 2 (S not positive definite) or 3 (S_jj <= 0).
template <int NC>
__device__ __forceinline__ int fx_norm_test(const KrylovArgs& a, const FxState<NC>& st, int n, int c, double& xsx) {
    const int nm = st.nm, RC = 3 * nm + 1;
    xsx = fx_red_get(fx_at<int>(st.v.red) + c * RC + nm + n, NC * RC) * fx_pow2(60 + st.bS[c]);
    if (n == 0) return xsx > 0.0 ? 0 : 3;
    const double w2 = xsx * fx_pow2(2 * st.we[c]), bound = a.breakdown_tol * a.breakdown_tol * st.hh[(n - 1) & 1][c];
    return w2 < -bound ? 2 : w2 > bound ? 0 : 1;
}

// The coefficients of column c for the update: integers, or in the lead FP64 in the place of h.
template <int NC>
__device__ __forceinline__ void fx_give_coefs(FxState<NC>& st, int n, int c, const double (&gk)[2]) {
    const int lane = threadIdx.x & 31;
    if (n >= st.lead) {
        fx_coefs(gk, n, fx_at<int2>(st.v.g) + c * st.nm, &st.q[c]);
        return;
    }
    __syncwarp();   // every lane has read h
    double* g = fx_at<double>(st.v.h) + c * st.nm;
    if (lane <= n) g[lane] = gk[0];
    if (lane + 32 <= n) g[lane + 32] = gk[1];
}

// First warp: S', the coefficients of the update, and the end of the column.
template <int NC>
__device__ __forceinline__ void fx_scalars(const KrylovArgs& a, FxState<NC>& st, int n, int c) {
    const int lane = threadIdx.x & 31, nm = st.nm, nu = st.nu, RC = 3 * nm + 1, RS = NC * RC, PK = nm * (nm + 1) / 2;
    const bool overlap = st.overlap;
    const int* red = fx_at<int>(st.v.red);
    const size_t col = (size_t)4 * (st.atom - a.atom_begin) + st.alpha0 + c;
    const int* rd = red + c * RC;
    double *f = fx_at<double>(st.v.f) + c * nm, *s = fx_at<double>(st.v.s) + c * nm, *h = fx_at<double>(st.v.h) + c * nm;
    const int bH = st.bH[c], bS = st.bS[c];
    double xsx;
    const int stop = fx_norm_test(a, st, n, c, xsx);
    if (stop) {
        if (lane == 0) {
            if (stop > 1) flag(a.status, stop == 2 ? DEV_NOT_SPD : DEV_ARG);
            st.nue[c] = n;
            st.done[c] = 1;
            atomicSub(&st.live, 1);
        }
    } else {
        const double fn = rsqrt(xsx), sn = fn * fx_pow2(60 + bS);
        if (lane == 0) {
            f[n] = fn;
            s[n] = sn;
        }
        double* hess = a.bstore ? a.bstore + (size_t)(4 * st.slot + st.alpha0 + c) * a.bstride + 3 * a.bvec : nullptr;
        if (hess && n > 0 && lane == 0)     // beta_(n-1) = |w|_S
            hess[(size_t)(n - 1) * nm + n] = sqrt(xsx * fx_pow2(2 * st.we[c])) *
                                             (f[n - 1] * fx_pow2(fx_at<int>(st.v.ex)[(NC + c) * nm + n - 1]));
        __syncwarp();
        double* E = fx_at<double>(st.v.E) + (size_t)c * PK;
        const int pk0 = n * (n + 1) / 2;
        bool big = false;
        for (int k = lane; k <= n; k += 32) {
            const double spk = f[k] * (sn * fx_red_get(rd + nm + k, RS));
            const double hk = s[k] * fx_red_get(rd + 2 * nm + k, RS);     // SU_k . H u_n over f 2^bH
            a.Sp[col * PK + pk0 + k] = spk;
            h[k] = hk;
            if (hess) hess[(size_t)n * nm + k] = hk * (fn * fx_pow2(bH));
            if (overlap) {
                const double e = k == n ? spk - 1.0 : spk;
                E[pk0 + k] = e;
                fx_at<float>(st.v.Ef)[(size_t)c * PK + pk0 + k] = (float)e;
                fx_at<float>(st.v.hf)[c * nm + k] = (float)hk;
                big |= (__double2hiint(e) & 0x7fffffff) >= (1023 - 40) << 20;
            }
        }
        if (__any_sync(0xffffffffu, big) && lane == 0) st.big[c] = 1;
        __syncwarp();
        if (n == nu - 1) {
            if (lane == 0) {
                st.done[c] = 1;
                atomicSub(&st.live, 1);
            }
        } else {
            // coefficients of the update in the integers' scales: f_k h_k, with both
            // passes' h_k - ((S' - I) h)_k where the second comes from S'
            double gk[2] = {0.0, 0.0};
            for (int r = 0; r < 2; ++r) {
                const int k = lane + 32 * r;
                if (32 * r > n) break;
                if (k > n) continue;
                double eh = 0.0;
                if (overlap && !st.big[c]) {
                    // entries of E below 2^-40 (Gram-Schmidt leaves 2^-48 or so): their product with h
                    // in single precision is within 64 x 2^-64 of h, far below the rounding of h itself
                    const float *Ef = fx_at<float>(st.v.Ef) + (size_t)c * PK, *hf = fx_at<float>(st.v.hf) + c * nm;
                    float e = 0.0f;
                    int at = k * (k + 1) / 2;          // row k up to the diagonal, then column k
                    for (int q = 0; q <= n; ++q) {
                        e = fmaf(Ef[at], hf[q], e);
                        at += q < k ? 1 : q + 1;
                    }
                    eh = (double)e;
                } else if (overlap) {
                    int at = k * (k + 1) / 2;
                    for (int q = 0; q <= n; ++q) {
                        eh = fma(E[at], h[q], eh);
                        at += q < k ? 1 : q + 1;
                    }
                }
                gk[r] = f[k] * (h[k] - eh);
            }
            fx_give_coefs(st, n, c, gk);
        }
    }
}

// Second warp: H', |P|^2, the exponents, and entry j of the vectors.
template <int NC>
__device__ __forceinline__ void fx_scalars_h(const KrylovArgs& a, FxState<NC>& st, int n, int c) {
    const int lane = threadIdx.x & 31, nm = st.nm, RC = 3 * nm + 1, RS = NC * RC, PK = nm * (nm + 1) / 2;
    const int* rd = fx_at<int>(st.v.red) + c * RC;
    const int bH = st.bH[c];
    double xsx;
    if (fx_norm_test(a, st, n, c, xsx)) return;
    const double fn = rsqrt(xsx), pn = fn * fx_pow2(60 + bH);
    const size_t col = (size_t)4 * (st.atom - a.atom_begin) + st.alpha0 + c;
    for (int k = lane; k <= n; k += 32) {
        const double fk = k == n ? fn : fx_at<double>(st.v.f)[c * nm + k];
        a.Hp[col * PK + n * (n + 1) / 2 + k] = fk * (pn * fx_red_get(rd + k, RS));
    }
    if (lane == 0) {
        st.hh[n & 1][c] = fx_red_get(rd + 3 * nm, RS) * 0x1p60;
        fx_at<int>(st.v.ex)[c * nm + n] = st.bS[c];
        fx_at<int>(st.v.ex)[(NC + c) * nm + n] = bH;
    }
    if (lane < 3) {
        const int al = st.alpha0 + c;
        const int4* w = fx_at<int4>(lane == 0 ? st.v.X : lane == 1 ? st.v.Y : st.v.P);
        fx_at<int2>(st.v.row)[(lane * NC + c) * nm + n] =
            reinterpret_cast<const int2*>(w + fx_unit<NC>(st.qJ, al >> 1, c))[al & 1];
    }
}

// w = P - sum_{k <= n} g_k X_k as 64-bit numbers, into X or in place (into P).
template <int NC, int T, int kMinB>
__device__ __forceinline__ void fx_update(FxState<NC>& st, int n, bool into_x, unsigned long long* bits) {
    const int tid = threadIdx.x, tc = tid % NC, units = st.units, upt = st.upt, kT = st.kT, kS = st.kS;
    const unsigned tm = FxTmem<T, kMinB>::base(st.tmem);
    const int4* P = fx_at<int4>(st.v.P);
    longlong2* W = fx_at<longlong2>(into_x ? st.v.X : st.v.P);
    const int2* g = fx_at<int2>(st.v.g) + tc * st.nm;
    const int q = st.q[tc];
    unsigned long long mW = 0;
#pragma unroll 1
    for (int i0 = 0; i0 < upt; i0 += 2) {
        Fx acc[4];
        const int ua = min(tid + i0 * T, units - 1), ub = min(tid + (i0 + 1) * T, units - 1);
        // vectors at to at + 3: w[kk], w[4 + kk] the two units of vector at + kk
        auto apply = [&](int at, int kend, const int4 (&w)[8]) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const int2 gk = at + kk < kend ? g[at + kk] : make_int2(0, 0);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    fx_mac(acc[2 * i], gk, fx_lo(w[4 * i + kk]));
                    fx_mac(acc[2 * i + 1], gk, fx_hi(w[4 * i + kk]));
                }
            }
        };
#pragma unroll 1
        for (int k = 0; k < kT && k <= n; k += 4) {
            int4 w[8];
            fx_tmem_ld4x2(tm + 4 * (k * upt + i0), 4 * upt, w);
            apply(k, n + 1, w);
        }
        auto sweep = [&](const int4* base, int k, int kend) {   // vectors k to kend - 1 at base
            const int4 *q = base, *const last = base + (size_t)(kend - 1 - k) * units;
            auto load = [&](int4 (&w)[8]) {   // past the end: the last vector again
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    w[kk] = q[ua];
                    w[4 + kk] = q[ub];
                    if (q < last) q += units;
                }
            };
            int4 wa[8], wb[8];
            load(wa);
#pragma unroll 1
            for (int at = k; at < kend; at += 8) {
                load(wb);
                apply(at, kend, wa);
                load(wa);
                if (at + 4 < kend) apply(at + 4, kend, wb);
            }
        };
        if (n >= kT) sweep(fx_at<int4>(st.v.cache), kT, min(kS, n + 1));
        if (n >= kS) sweep(st.gU + (size_t)kS * units, kS, n + 1);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int u = tid + (i0 + i) * T;
            if (i0 + i < upt && u < units) {
                const int4 p = P[u];
                longlong2 w;
                w.x = fx_shr(((long long)p.x << 28) + p.y, q) - fx_fold(acc[2 * i]);
                w.y = fx_shr(((long long)p.z << 28) + p.w, q) - fx_fold(acc[2 * i + 1]);
                mW |= fx_abs_bits(w.x) | fx_abs_bits(w.y);
                W[u] = w;
            }
        }
        __syncwarp();
    }
    if (st.done[tc]) mW = 0;
    __syncwarp();
    fx_or<NC>(mW, bits + tc);
}

// The same in the lead, in FP64: w = 2^sP h - sum_{k <= n} g_k u_k, h and u_k as FP64.
template <int NC, int T>
__device__ __forceinline__ void fx_update_lead(FxState<NC>& st, int n, bool into_x, unsigned* top) {
    const int tid = threadIdx.x, tc = tid % NC, units = st.units;
    double2* W = fx_at<double2>(into_x ? st.v.X : st.v.P);
    const double* g = fx_at<double>(st.v.h) + tc * st.nm;
    const double fh = fx_pow2(st.sP[tc]);
    unsigned mT = 0;
#pragma unroll 1
    for (int u = tid; u < units; u += T) {
        double2 w = st.hd[u];
        w.x *= fh;
        w.y *= fh;
        const double2* q = st.gD + u;
#pragma unroll 4
        for (int k = 0; k <= n; ++k, q += units) {
            const double2 v = *q;
            w.x = fma(-g[k], v.x, w.x);
            w.y = fma(-g[k], v.y, w.y);
        }
        mT = max(mT, max(fx_top(w.x), fx_top(w.y)));
        W[u] = w;
    }
    if (st.done[tc]) mT = 0;
    __syncwarp();
    fx_max<NC>(mT, top + tc);
}

// Where vector k of U lives outside tensor memory.
template <int NC>
__device__ __forceinline__ int4* fx_ubase(const FxState<NC>& st, int k) {
    return k < st.kS ? fx_at<int4>(st.v.cache) + (k - st.kT) * st.units : st.gU + (size_t)k * st.units;
}

// u_1 = e_j, unscaled, for the columns st.alpha0 to + NC - 1, and an empty column state.
template <int NC, int T, int kMinB>
__device__ __forceinline__ void fx_start(FxState<NC>& st) {
    const int tid = threadIdx.x, units = st.units, upt = st.upt, red_words = 3 * NC * (3 * st.nm + 1);
    int4* X = fx_at<int4>(st.v.X);
    for (int u = tid; u < units; u += T) {
        X[u] = make_int4(0, 0, 0, 0);
        st.gD[u] = make_double2(0.0, 0.0);
        if (st.xa) st.xa[u] = make_double2(0.0, 0.0);
    }
    for (int q = tid; q < red_words; q += T) fx_at<int>(st.v.red)[q] = 0;
    if (tid < NC) {
        st.bits[0][tid] = st.bits[1][tid] = 0;
        st.top[0][tid] = st.top[1][tid] = 0;
        st.done[tid] = st.big[tid] = st.q[tid] = 0;
        st.nue[tid] = st.nu;
    }
    if (tid == 0) {
        st.live = NC;
        st.lead = kLead;
        st.small = 0;
    }
    __syncthreads();
    if (tid < NC) {
        const int al = st.alpha0 + tid, at = fx_unit<NC>(st.qJ, al >> 1, tid);
        reinterpret_cast<int*>(X + at)[2 * (al & 1)] = 1 << 28;
        reinterpret_cast<double*>(st.gD + at)[al & 1] = 0x1p56;
        if (st.xa) reinterpret_cast<double*>(st.xa + at)[al & 1] = 0x1p56;
    }
    __syncthreads();
    const unsigned tm = FxTmem<T, kMinB>::base(st.tmem);
    for (int i = 0; i < upt; ++i) {
        const int u = tid + i * T;
        const int4 w = u < units ? X[u] : make_int4(0, 0, 0, 0);
        if (st.kT > 0) fx_tmem_st(tm + 4 * i, w);
        else if (u < units) fx_ubase(st, 0)[u] = w;
    }
}

// H X and S X (64-bit sums in P and Y, FP64 in the lead) into split form; S X_n also into the basis SU.
template <int NC, int T>
__device__ __forceinline__ void fx_take_products(FxState<NC>& st, int n) {
    const int tid = threadIdx.x, tc = tid % NC, units = st.units;
    int4 *P = fx_at<int4>(st.v.P), *Y = fx_at<int4>(st.v.Y);
    int4* yn = n < st.kY ? fx_at<int4>(st.v.cache) + (st.kS - st.kT + n) * units : st.gY + (size_t)n * units;
    if (n < st.lead) {
        const int sH = fx_lead_shift(st.top[0][tc]), sS = fx_lead_shift(st.top[1][tc]);
        const double fH = fx_pow2(sH), fS = fx_pow2(sS);
        for (int u = tid; u < units; u += T) {
            const double2 h = reinterpret_cast<const double2*>(P)[u];
            st.hd[u] = h;
            P[u] = fx_lead_split(h, fH);
            const int4 y = fx_lead_split(reinterpret_cast<const double2*>(Y)[u], fS);
            Y[u] = y;
            yn[u] = y;
        }
        if (tid < NC) {
            st.sP[tid] = sH;
            st.bH[tid] = -sH;
            st.bS[tid] = -sS;
        }
    } else {
        const int shH = fx_shift(st.bits[0][tc]), shS = fx_shift(st.bits[1][tc]);
        for (int u = tid; u < units; u += T) {
            P[u] = fx_norm2(reinterpret_cast<const longlong2*>(P)[u], shH);
            const int4 y = fx_norm2(reinterpret_cast<const longlong2*>(Y)[u], shS);
            Y[u] = y;
            yn[u] = y;
        }
        if (tid < NC) {
            st.bH[tid] = 56 - st.sc.eH + shH;
            st.bS[tid] = 56 - st.sc.eS + shS;
        }
    }
    __syncwarp();
}

// w (64-bit numbers in X; FP64 in the lead, sh then the power of two it is multiplied by) becomes
// X_(n+1), in X and in the basis. The lead goes on while an atom that is reached stays below 2^-kSmall of
// the largest in the last two vectors.
template <int NC, int T, int kMinB>
__device__ __forceinline__ void fx_take_vector(FxState<NC>& st, int n, int sh) {
    const int tid = threadIdx.x, units = st.units, upt = st.upt;
    const bool dead = st.done[tid % NC] != 0, in_lead = n < st.lead;
    int4* X = fx_at<int4>(st.v.X);
    const double lead = fx_pow2(sh);
    const unsigned tm = FxTmem<T, kMinB>::base(st.tmem);
    double2* const D = st.gD + (size_t)n * units;
    bool small = false;
    for (int i = 0; i < upt; ++i) {
        const int u = tid + i * T;
        int4 w = make_int4(0, 0, 0, 0);
        if (in_lead) {
            unsigned top = 0;
            if (u < units) {
                double2 wd = make_double2(0.0, 0.0);
                if (!dead) wd = reinterpret_cast<const double2*>(X)[u];
                wd.x *= lead;
                wd.y *= lead;
                if (n + 1 >= kLead) {
                    const double2 before = D[u];
                    top = max(max(fx_top(wd.x), fx_top(wd.y)), max(fx_top(before.x), fx_top(before.y)));
                }
                D[units + u] = wd;
                if (st.xa && n + 1 <= kLead) st.xa[u] = wd;
                w = fx_lead_split(wd, 1.0);
                X[u] = w;
            }
            __syncwarp();
            if (n + 1 >= kLead) {   // an atom's other two orbitals are NC lanes on
                top = max(top, __shfl_xor_sync(0xffffffffu, top, NC));
                small |= !dead && top > 0u && top < (unsigned)(1023 + 56 - kSmall) << 20;
            }
        } else if (u < units) {
            if (!dead) w = fx_norm2(reinterpret_cast<const longlong2*>(X)[u], sh);
            X[u] = w;
        }
        if (n + 1 < st.kT) fx_tmem_st(tm + 4 * ((n + 1) * upt + i), w);
        else if (u < units) fx_ubase(st, n + 1)[u] = w;
    }
    if (small) st.small = 1;
}

// The second classical pass between its two updates: w (64-bit numbers in P) into split form, its
// products with SU and the coefficients from them. Every thread of the CTA calls it.
template <int NC, int T>
__device__ __forceinline__ void fx_second_coefs(FxState<NC>& st, int n, int sh) {
    const int tid = threadIdx.x, c = tid >> 5, lane = tid & 31, nm = st.nm, RC = 3 * nm + 1, RS = NC * RC;
    int4* P = fx_at<int4>(st.v.P);
    int* red = fx_at<int>(st.v.red);
    if (n < st.lead) {
        const double lead = fx_pow2(sh);
        for (int u = tid; u < st.units; u += T) {
            const double2 wd = reinterpret_cast<const double2*>(P)[u];
            st.hd[u] = wd;
            P[u] = fx_lead_split(wd, lead);
        }
        if (tid < NC) st.sP[tid] = sh;
    } else {
        for (int u = tid; u < st.units; u += T) P[u] = fx_norm2(reinterpret_cast<const longlong2*>(P)[u], sh);
    }
    __syncwarp();
    fx_sweep_y<NC, T>(st, n, 0);
    __syncthreads();
    if (c < NC && !st.done[c]) {
        double gk[2] = {0.0, 0.0};
        for (int r = 0; r < 2; ++r) {
            const int k = lane + 32 * r;
            if (k <= n)
                gk[r] = fx_at<double>(st.v.f)[c * nm + k] * (fx_at<double>(st.v.s)[c * nm + k] * fx_red_get(red + c * RC + k, RS));
        }
        fx_give_coefs(st, n, c, gk);
    }
    __syncthreads();
    for (int q = tid; q < 3 * RS; q += T) red[q] = 0;
    __syncthreads();
}

// Kept bases (KrylovArgs::bstore): u_n, S u_n and H u_n of the live columns in FP64, at the exact
// gradient's positions (zero where a position holds no atom).
template <int NC, int T>
__device__ __forceinline__ void fx_keep_step(const KrylovArgs& a, FxState<NC>& st, int n) {
    const int np = (st.n_at + 31) / 32 * 32, nm = st.nm;
    const int* pos_atom = fx_at<int>(st.v.pos_atom);
    for (int q = threadIdx.x; q < np * 4 * NC; q += T) {
        const int r = q & 3, p = (q >> 2) % np, c = (q >> 2) / np, at = pos_atom[p];
        if (n >= st.nue[c]) continue;
        double* out = a.bstore + (size_t)(4 * st.slot + st.alpha0 + c) * a.bstride + (size_t)n * np * 4 + 4 * p + r;
        double u = 0.0, su = 0.0, hu = 0.0;
        if (at >= 0) {
            const int k = 2 * fx_unit<NC>(at, r >> 1, c) + (r & 1);
            const double f = fx_at<double>(st.v.f)[c * nm + n];
            u = f * fx_value(fx_at<int2>(st.v.X)[k]);
            su = f * fx_pow2(fx_at<int>(st.v.ex)[c * nm + n]) * fx_value(fx_at<int2>(st.v.Y)[k]);
            hu = f * fx_pow2(fx_at<int>(st.v.ex)[(NC + c) * nm + n]) * fx_value(fx_at<int2>(st.v.P)[k]);
        }
        out[0] = u;
        out[a.bvec] = su;
        out[2 * a.bvec] = hu;
    }
}

// Results of the NC columns: nu_eff, row j of U, SU and HU, the pattern rows of U. The vectors in
// tensor memory pass through the work arrays X and P, which are free here, two at a time.
template <int NC, int T, int kMinB>
__device__ __forceinline__ void fx_results(const KrylovArgs& a, FxState<NC>& st, int J) {
    const int tid = threadIdx.x, nm = st.nm, nu = st.nu, units = st.units, upt = st.upt, kT = st.kT, alpha0 = st.alpha0;
    const size_t col0 = (size_t)4 * (J - a.atom_begin) + alpha0;
    const double* f = fx_at<double>(st.v.f);
    int4 *X = fx_at<int4>(st.v.X), *P = fx_at<int4>(st.v.P);
    if (tid < NC) {
        const int ne = st.nue[tid];
        a.nu_eff[4 * J + alpha0 + tid] = ne;
        if (ne < nu && !a.again) flag(a.status, DEV_BREAKDOWN);
        if (a.flops) atomicAdd(a.flops, column_flops(a, st.n_at, st.nent, ne, st.overlap));
    }
    for (int q = tid; q < 3 * NC * nm; q += T) {
        const int n = q % nm, t = q / nm, c = t % NC, kind = t / NC;
        if (n >= st.nue[c]) continue;
        double* out = kind == 0 ? a.urow : kind == 1 ? a.surow : a.hurow;
        const double w = fx_value(fx_at<int2>(st.v.row)[q]) * f[c * nm + n];
        out[(col0 + c) * nm + n] = kind == 0 ? w : w * fx_pow2(fx_at<int>(st.v.ex)[((kind - 1) * NC + c) * nm + n]);
    }
    if (a.bstore) {   // H' beside the kept bases
        const int PK = nm * (nm + 1) / 2;
        for (int q = tid; q < NC * PK; q += T) {
            const int c = q / PK, k = q % PK;
            a.bstore[(size_t)(4 * st.slot + alpha0 + c) * a.bstride + 3 * a.bvec + (size_t)nm * nm + k] = a.Hp[(col0 + c) * PK + k];
        }
    }
    if (a.UP) {
        const int e0 = a.row_ptr[J], rows = 4 * (a.row_ptr[J + 1] - e0);
        auto put = [&](int q, int k, const int4* uk) {
            const int c = q % NC, er = q / NC, r = er & 3;
            if (k >= st.nue[c]) return;
            const int2 w = reinterpret_cast<const int2*>(uk + fx_unit<NC>(fx_at<short>(st.v.at)[er >> 2], r >> 1, c))[r & 1];
            a.UP[((size_t)((e0 + (er >> 2) - a.up_block0) * 4 + alpha0 + c) * 4 + r) * nm + k] = f[c * nm + k] * fx_value(w);
        };
        const unsigned tm = FxTmem<T, kMinB>::base(st.tmem);
        __syncthreads();
        for (int k = 0; k < kT; k += 2) {
            for (int i = 0; i < upt; ++i) {
                int4 w[2];
                fx_tmem_ld<2>(tm + 4 * (k * upt + i), 4 * upt, w);
                const int u = tid + i * T;
                if (u < units) {
                    X[u] = w[0];
                    P[u] = w[1];
                }
            }
            __syncthreads();
            for (int q = tid; q < rows * NC * 2; q += T) put(q >> 1, k + (q & 1), (q & 1) ? P : X);
            __syncthreads();
        }
        for (int q = tid; q < rows * NC * (nu - kT); q += T) {
            const int k = kT + q % (nu - kT);
            put(q / (nu - kT), k, fx_ubase(st, k));
        }
    }
    __syncthreads();
}

// kDense: caller matrices (dense blocks) instead of two-centre ones.
template <int NC, int T, int kMinB, bool kDense>
__global__ void __launch_bounds__(T, kMinB) k_krylov_fixed(const __grid_constant__ KrylovArgs a, const __grid_constant__ FxArgs x) {
    __shared__ FxState<NC> st;
    if (!x.scale->ok) return;   // (caller matrices: the FP64 kernel takes them)
    using Tm = FxTmem<T, kMinB>;
    if (threadIdx.x == 0) {
        const size_t cta_units = (size_t)a.nu_max * a.na_max * 2 * NC;
        st.v = fx_layout<NC, T>(a.na_max, a.nu_max, a.deg_max + 1, a.reorth != 0, a.bstore != nullptr);
        st.sc = *x.scale;
        st.rec = x.rec;
        st.gU = reinterpret_cast<int4*>(a.scratch) + (3 * cta_units + (size_t)a.na_max * 2 * NC) * blockIdx.x;
        st.gY = st.gU + cta_units;
        st.gD = reinterpret_cast<double2*>(st.gY + cta_units);
        st.hd = st.gD + cta_units;
        st.Es = x.Es;
        st.Ep = x.Ep;
        st.nm = a.nu_max;
        st.overlap = a.reorth != 0;
    }
    if (threadIdx.x < 32) fx_tmem_alloc(&st.tmem, Tm::cols);
    __syncthreads();

    for (int iter = 0;; ++iter) {
        if (threadIdx.x == 0) {
            const int item = a.queue ? atomicAdd(a.queue, 1) : blockIdx.x + iter * gridDim.x;
            const int idx = x.split ? item / (4 / NC) : item;
            int J = idx < a.n_items ? a.order[idx] : -1;
            if (a.again && J >= 0 && (J < a.only_lo || J >= a.only_hi)) J = -2;
            st.atom = J;
            st.slot = a.again ? idx : J;
            st.alpha0 = x.split ? item % (4 / NC) * NC : 0;
            st.nent = 0;
            if (J >= 0) {
                const int n_at = a.cl_ptr ? a.cl_ptr[J + 1] - a.cl_ptr[J] : a.n_atoms;
                const int units = n_at * 2 * NC, upt = (units + T - 1) / T, nu = min(nu_for(a, n_at), a.nu_max);
                const int vecs = (int)((x.smem_bytes - st.v.cache) / sizeof(int4)) / units;   // that fit in shared memory
                st.n_at = n_at;
                st.units = units;
                st.upt = upt;
                st.nu = nu;
                // (the update reads up to one unit past a vector in tensor memory)
                st.kT = min((Tm::units - 1) / upt, nu) & ~3;
                st.kS = st.kT + min(nu - st.kT, vecs);
                st.kY = min(nu, vecs - (st.kS - st.kT));
                // the last vector's place in shared memory while that is free
                st.xa = st.kS > st.kT && st.kS - 1 > kLead
                            ? reinterpret_cast<double2*>(fx_at<int4>(st.v.cache) + (st.kS - 1 - st.kT) * units) : nullptr;
            }
        }
        __syncthreads();
        const int J = st.atom;
        if (J == -1) break;
        if (J < 0) {
            __syncthreads();
            continue;
        }
        if (st.n_at > a.na_max) {
            if (threadIdx.x == 0) flag(a.status, DEV_CAPACITY);
            __syncthreads();
            continue;
        }
        fx_view<NC, T, kDense>(a, st, J, a.cl_ptr ? a.cl_ptr[J] : 0, st.n_at);
        if (a.bstore)
            balanced_positions<32, T>(st.n_at, (st.n_at + 31) / 32, fx_at<int>(st.v.deg), fx_at<int>(st.v.pos),
                                      fx_at<int>(st.v.pos_atom));
        for (;;) {
            fx_start<NC, T, kMinB>(st);
            const int nu = st.nu;
            for (int n = 0; n < nu; ++n) {
                const bool lead = n < st.lead;
                if (lead) fx_products_lead<NC, T, kDense>(a, st, n);
                else if constexpr (kDense) fx_products_dense<NC, T>(st);
                else fx_products<NC, T>(st);
                __syncthreads();
                fx_take_products<NC, T>(st, n);
                fx_pass_a<NC, T, kMinB>(st, n);
                const int warp = threadIdx.x >> 5;
                const bool idle = warp >= 2 * NC || st.done[warp % NC];   // (done changes below)
                __syncthreads();
                // the magnitudes were last read before pass A; the update's, of every warp, come after
                // the barrier below
                if (threadIdx.x < NC) {
                    st.bits[0][threadIdx.x] = st.bits[1][threadIdx.x] = 0;
                    st.top[0][threadIdx.x] = st.top[1][threadIdx.x] = 0;
                }
                if (!idle && warp < NC) fx_scalars<NC>(a, st, n, warp);
                else if (!idle) fx_scalars_h<NC>(a, st, n, warp - NC);
                __syncthreads();
                if (a.bstore) {
                    fx_keep_step<NC, T>(a, st, n);
                    __syncthreads();
                }
                for (int q = threadIdx.x; q < 3 * NC * (3 * st.nm + 1); q += T) fx_at<int>(st.v.red)[q] = 0;
                if (threadIdx.x < NC) st.we[threadIdx.x] = 0;   // read and written by this thread until the next step
                if (st.live == 0) {
                    __syncthreads();   // st.live is set again for the next columns
                    break;
                }
                for (int pass = st.overlap ? 1 : 0; pass < 2; ++pass) {
                    if (lead) fx_update_lead<NC, T>(st, n, pass == 1, st.top[pass]);
                    else fx_update<NC, T, kMinB>(st, n, pass == 1, st.bits[pass]);
                    __syncthreads();
                    const int tc = threadIdx.x % NC;
                    const int sh = lead ? fx_lead_shift(st.top[pass][tc]) : fx_shift(st.bits[pass][tc]);
                    if (threadIdx.x < NC) st.we[tc] += lead ? -sh : st.q[tc] + sh;   // P = 2^we (the new integers)
                    if (pass == 1) fx_take_vector<NC, T, kMinB>(st, n, sh);
                    else fx_second_coefs<NC, T>(st, n, sh);
                }
                __syncthreads();
                if (threadIdx.x < NC) {
                    st.bits[0][threadIdx.x] = st.bits[1][threadIdx.x] = 0;
                    st.top[0][threadIdx.x] = st.top[1][threadIdx.x] = 0;
                }
                if (threadIdx.x == 0) {
                    if (st.small) st.lead = max(st.lead, n + 2);
                    st.small = 0;
                }
                __syncthreads();
            }
            __syncthreads();
            fx_results<NC, T, kMinB>(a, st, J);
            const int next = st.alpha0 + NC;
            __syncthreads();
            if (x.split || next >= 4) break;
            if (threadIdx.x == 0) st.alpha0 = next;
            __syncthreads();
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) fx_tmem_free(st.tmem, Tm::cols);
}

namespace {
struct FxForm {
    int nc, t, min_b;       // columns at a time, threads, CTAs an SM holds
    const void *fn, *fn_dense;
    FxLayout (*layout)(int, int, int, bool, bool);
};
template <int NC, int T, int B>
FxForm fx_form() { return {NC, T, B, reinterpret_cast<const void*>(&k_krylov_fixed<NC, T, B, false>),
            reinterpret_cast<const void*>(&k_krylov_fixed<NC, T, B, true>), &fx_layout<NC, T>}; }
const FxForm kForms[] = {fx_form<4, 384, 1>(), fx_form<1, 128, 2>()};
constexpr int kMaxUpt = 7;      // units of a thread: eight lanes' sums of 2 x 7 products of 2^112 / 2^56 stay below 2^63
constexpr size_t kSmemSM = 233472, kSmemCta = 232448;   // per SM, and the most one CTA may have
constexpr size_t kSmemStatic = 2048;                    // bound on the kernel's static shared memory

size_t form_bytes(const FxForm& f, int na, int max_row, int nu, bool overlap, bool store) {
    return f.layout(na, nu, max_row, overlap, store).cache;
}
}  // namespace

// The form for a system of n atoms: all four columns of an atom in one CTA of 384 threads, or,
// while that leaves SMs idle, one column per CTA of 128 threads, two of them to an SM. The second
// takes 1.3 times the first's time per column when both fill the chip (4096-atom diamond: 42.0
// against 33.0 ms) but spreads an atom's columns over up to four SMs: the smaller number of
// column times in whole waves decides (64 atoms: 2.6 against 4; 211: 7.8 against 8). By the
// system's size alone, not by the class or the batch: the two forms round their partial sums
// differently, and results do not depend on the batches.
int fx_form_for(int n, int sms) {
    const double one = 4.0 * ((n + sms - 1) / sms), split = 1.3 * 2.0 * ((4LL * n + 2 * sms - 1) / (2 * sms));
    return split < one ? 1 : 0;
}

int fx_blocks_per_sm(int form, int na, int max_row, int nu, bool overlap, bool store) {
    const FxForm& f = kForms[form];
    if (na * 2 * f.nc > kMaxUpt * f.t) return 0;
    const size_t b = form_bytes(f, na, max_row, nu, overlap, store) + kSmemStatic;
    if (b > kSmemCta) return 0;
    return std::min<int>(f.min_b, (int)(kSmemSM / (b + 1024)));   // registers and tensor memory: min_b
}

int fx_items(int form, int count) { return count * (4 / kForms[form].nc); }

size_t fx_scratch_doubles(int form, int nu, int na) { return ((size_t)3 * nu + 1) * na * 4 * kForms[form].nc; }

void fx_columns(const KrylovArgs& a, FxArgs x, int form, int grid, int ctas_per_sm, cudaStream_t st) {
    const FxForm& f = kForms[form];
    // the shared memory of an SM split over its CTAs; what the work arrays leave holds basis vectors
    const size_t all = form_bytes(f, a.na_max, a.deg_max + 1, a.nu_max, a.reorth != 0, a.bstore != nullptr) +
                       2 * sizeof(int4) * (size_t)a.nu_max * a.na_max * 2 * f.nc;
    const size_t share = std::min(kSmemCta, kSmemSM / ctas_per_sm - 1024) - kSmemStatic;
    x.smem_bytes = (int)(std::min(all, share) & ~(size_t)15);
    x.split = f.nc < 4;
    const void* fn = a.skr ? f.fn : f.fn_dense;
    smem_at_least(fn, kSmemCta - kSmemStatic);   // what any launch of it may ask for
    void* args[] = {const_cast<KrylovArgs*>(&a), &x};
    cudaLaunchKernel(fn, dim3(grid), dim3(f.t), args, (size_t)x.smem_bytes, st);
}

}  // namespace elses
