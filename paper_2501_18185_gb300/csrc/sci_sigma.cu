// libsci hot path: sigma = H c (Sec. 2.4, the diagonalisation paragraph).
//
// sigma_I = H_II c_I + sum_{J single of I} H_IJ c_J + sum_{J double of I} H_IJ c_J,
// each off-diagonal element evaluated on the fly from the two occupation strings by the
// Slater-Condon rules (Sec. 2.3: matrix-element categories with 0, 1, 2 differences).
//
// Connection finding is done once at setup by bucketing: two determinants are within a
// double excitation exactly when they share an (N-2)-electron sub-string K, and they
// share exactly one such K when they differ by a double excitation.  So the doubles of
// the whole space are the disjoint pairs inside the buckets of equal K.  For a bra
// I = K + {a,b} and a ket J = K + {i,j} (a<b, i<j):
//     H_IJ = (-1)^(pi_I + pi_J) [(ai|bj) - (aj|bi)],
//     pi_X = #(K below x) + #(K below y) for the extras {x,y} of X,
// since applying a_j, a_i, a+_a, a+_b to J passes pi_J + pi_I + 2 occupied orbitals.
// Singles are the pairs inside the buckets of equal (N-1)-electron S:
//     H_IJ = (-1)^(pi_I + pi_J) [h_ai + sum_{k in S} ((ai|kk) - (ak|ki))],
// evaluated as F^ref_ai plus the terms of the orbitals where S and the reference differ
// (the closed-shell reference simplification of Sec. 2.3).
//
// Kernel shape (bucket-major, no tensor cores: this is a sparse gather).  A CTA owns
// the whole buckets that start in its range of table rows (its window), and stages every
// member of them in shared memory: the member's ket code, its ket offset into the
// pair-integral table and its coefficients pre-multiplied by (-1)^pi.  A thread takes a row
// and the members of its bucket that are doubles of it; the table stores bra indices
// fastest, so lanes that share a bucket read nearby entries.  A row's partial sum is added
// to sigma with one FP64 atomic add per (bucket, member).  Three things bound it, in turn:
// the FP64 pipe (2 FMA per clock per SM: a warp instruction holds it 16 cycles whatever its
// active lanes), the L1's rate of scattered accesses and the latency of the L2 gathers.
// Buckets are handled by size (launch_doubles): above the tile threshold by
// k_doubles_tiled, 256 members of one bucket as the rows of a CTA and the bucket streamed
// through shared memory; then by k_doubles_aligned (lanes of a bucket in step) or
// k_doubles_sorted (rows sorted by their number of doubles, lanes on useful products only);
// the smallest by k_doubles_small, in registers.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "sci_bucket.cuh"
#include "sci_ds.cuh"
#include "sci_internal.cuh"

using sci::zdbl;

#define SCI_CK(call)                                                 \
    do {                                                             \
        int _rc = sci_cuda_check(ctx, (call), #call);                \
        if (_rc != SCI_OK) return _rc;                               \
    } while (0)

namespace {

// ------------------------------------------------------------------ scalar ops
// Sign flips are integer XORs of the sign bit: on GB300 the FP64 pipe is the scarce
// resource (1.2 TFLOP/s), so no FP64 instruction is spent on a negation.
__device__ __forceinline__ double flip(bool f, double a)
{
    return __longlong_as_double(__double_as_longlong(a) ^ ((unsigned long long)f << 63));
}
__device__ __forceinline__ float flip(bool f, float a) { return __int_as_float(__float_as_int(a) ^ ((int)f << 31)); }
__device__ __forceinline__ zdbl flip(bool f, zdbl a) { return zdbl{flip(f, a.x), flip(f, a.y)}; }
__device__ __forceinline__ float2 flip(bool f, float2 a) { return make_float2(flip(f, a.x), flip(f, a.y)); }
__device__ __forceinline__ float4 flip(bool f, float4 a)
{
    return make_float4(flip(f, a.x), flip(f, a.y), flip(f, a.z), flip(f, a.w));
}

__device__ __forceinline__ void zero(double &a) { a = 0.0; }
__device__ __forceinline__ void zero(zdbl &a) { a = zdbl{0.0, 0.0}; }

// acc += t * c
__device__ __forceinline__ void fma_acc(double &acc, double t, double c) { acc = fma(t, c, acc); }
__device__ __forceinline__ void fma_acc(zdbl &acc, zdbl t, zdbl c)
{
    acc.x = fma(t.x, c.x, acc.x);
    acc.x = fma(-t.y, c.y, acc.x);
    acc.y = fma(t.x, c.y, acc.y);
    acc.y = fma(t.y, c.x, acc.y);
}

__device__ __forceinline__ void red_add(double *p, double v) { atomicAdd(p, v); }
__device__ __forceinline__ void red_add(zdbl *p, zdbl v)
{
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}
// The same, not sent when the sum is zero (rows whose bucket holds only single
// excitations of them sum to exactly 0, and adding +-0 leaves sigma unchanged).  The
// test reads the bits on the integer pipe.  Used where the atomics are the bound (FP32
// storage at several vectors: -4% there); elsewhere the branch costs more than it saves.
__device__ __forceinline__ void red_add_nz(double *p, double v)
{
    if ((__double_as_longlong(v) << 1) != 0) atomicAdd(p, v);
}

template <typename T> __device__ __forceinline__ T ldg(const T *p) { return __ldg(p); }
template <> __device__ __forceinline__ zdbl ldg<zdbl>(const zdbl *p)
{
    double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return zdbl{v.x, v.y};
}

using sci::col_code;
using sci::kSmallBucket;
using sci::kSortBucket;
using sci::disjoint;
using sci::doubles_mask;
using sci::row_code;
using sci::window;

// acc type for a storage type
template <typename TS> struct AccOf { using type = double; };
template <> struct AccOf<zdbl> { using type = zdbl; };

constexpr int kThreads = 256;
constexpr int kUnroll = 4;
// Rows per CTA.  Eight 256-thread CTAs fit an SM; what shared memory leaves of the
// 256 KB L1 for caching decides the speed (measured on the 2M-determinant space:
// 5.20 ms at 768 rows, 5.34 at 1024, 7.63 at 1280, where L1 is nearly gone).
constexpr int kRowsPerCta = 768;
// The FP32-storage kernel at 8 vectors (the mixed Davidson's block) stages 40 bytes per
// window row, so its window rows and its CTAs per SM (registers) are set apart.  Measured
// on the 2M-determinant space (doubles kernel, 8 vectors): 768 rows at 64 registers (4
// CTAs/SM by shared memory and registers) 15.84 ms; 512 rows at 5 CTAs/SM (48 registers,
// no spills) 14.88 ms; 448 rows at 6 (40 registers) 15.17 ms; 384 rows 15.57 ms.
#ifndef SCI_F32_ROWS
#define SCI_F32_ROWS 512
#endif
#ifndef SCI_F32_MINB
#define SCI_F32_MINB 5
#endif

// ------------------------------------------------------------------ row ranges
// A RANGED launch walks the range tables of sci_set_row_range() and computes only the
// members whose determinant lies in [rr.rb, rr.re).  Its CTA lists those rows of its
// window, in window order, in shared memory (a ballot per warp and a prefix over the
// warps), so that the lanes of a warp still own neighbouring rows of equal-size buckets;
// a window with no such row returns before staging anything.  Returns the row count.
__device__ __forceinline__ int owned_rows(const uint32_t *__restrict__ e_idx, int64_t r0, int W, sci::RowRange rr,
                                          uint16_t *s_own)
{
    __shared__ int s_wcnt[kThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int total = 0;
    for (int base = 0; base < W; base += blockDim.x) {
        const int q = base + (int)threadIdx.x;
        bool own = false;
        if (q < W) {
            const int64_t I = e_idx[r0 + q];
            own = I >= rr.rb && I < rr.re;
        }
        const unsigned m = __ballot_sync(0xffffffffu, own);
        if (lane == 0) s_wcnt[wid] = __popc(m);
        __syncthreads();
        int off = total, tot = total;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            const int c = s_wcnt[w];
            off += w < wid ? c : 0;
            tot += c;
        }
        if (own) s_own[off + __popc(m & ((1u << lane) - 1u))] = (uint16_t)q;
        total = tot;
        __syncthreads();
    }
    return total;
}

// ------------------------------------------------------------------ sigma = diag * c
// rows [row0, row0 + nrows) of S = H_II C
template <typename TC, typename TA>
__global__ void k_sigma_init(const double *__restrict__ hdiag, const TC *__restrict__ C, TA *__restrict__ S,
                             int64_t row0, int64_t nrows, int nvec)
{
    const int64_t total = nrows * nvec;
    C += row0 * nvec;
    S += row0 * nvec;
    hdiag += row0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        double h = hdiag[t / nvec];
        TA s;
        zero(s);
        if constexpr (sizeof(TC) == sizeof(zdbl)) {
            zdbl c = C[t];
            s = TA{h * c.x, h * c.y};
        } else {
            s = (TA)(h * (double)C[t]);
        }
        S[t] = s;
    }
}

// ------------------------------------------------------------------ doubles, paired FP32
// The same bucket walk with the products and per-row sums in "double-single" arithmetic
// on the FP32 pipes: an FP64 value x is carried as hi + lo with hi = fl32(x) and
// lo = fl32(x - hi).  For t = th + tl and c = ch + cl the product is
//     p = fl(th*ch),  e = (th*ch - p) + th*cl + tl*ch      (exact first term via FMA;
// the dropped tl*cl is ~2^-48 of |tc|), and the sum (hi, lo) takes p by TwoSum
// (Knuth) with e and the rounding error folded into lo.  lo is renormalised into hi every
// kUnroll pairs.  The row sum leaves the kernel as fp64(hi) + fp64(lo) through the same
// FP64 atomic add as the FP64 path.
using sci::Ds;
using sci::ds_fma;
using sci::ds_renorm;
using sci::ds_value;
using sci::ds_zero;
using sci::f2d_int;

__device__ __forceinline__ float2 ds_split(double x)
{
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
}

__device__ __forceinline__ float2 ds_split(float x) { return make_float2(x, 0.f); }

// split the vector group C[:, v0:v0+G] into paired floats, once per sigma call (so the
// staging in the bucket kernel, which touches each coefficient many times, only copies)
template <typename TC>
__global__ void k_split_c(const TC *__restrict__ C, int64_t M, int nvec, int v0, int G, float2 *__restrict__ out)
{
    const int64_t total = M * G;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x)
        out[t] = ds_split(C[(t / G) * nvec + v0 + t % G]);
}

// a += t * c for FP32 t and c: the product is exact as p + e (e by FMA), the sum is
// compensated as in ds_fma
__device__ __forceinline__ void ds_fma1(Ds &a, float t, float c)
{
    const float p = t * c;
    const float e = fmaf(t, c, -p);
    const float s = a.hi + p;
    const float bv = s - a.hi;
    const float err = (a.hi - (s - bv)) + (p - bv);
    a.lo += err + e;
    a.hi = s;
}

__global__ void k_split_cz(const zdbl *__restrict__ C, int64_t M, int nvec, int v0, int G, float4 *__restrict__ out)
{
    const int64_t total = M * G;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const zdbl c = C[(t / G) * nvec + v0 + t % G];
        const float2 re = ds_split(c.x), im = ds_split(c.y);
        out[t] = make_float4(re.x, re.y, im.x, im.y);
    }
}

// ------------------------------------------------------------------ chained launches
// The doubles launches of one vector group, and in FP64 those of all groups and the singles,
// only read what was complete before the first of them and add into sigma (or store to slots
// of their own), so each may start while its predecessor drains: a dependent launch
// (programmatic stream serialization) begins once every CTA of the predecessor has started
// and executed chain_next().  A later launch must still see all of them complete, so a launch
// completes only after its predecessor: its last CTA (the singles: every CTA, at its end) does
// nothing but wait for it.  A selected space takes seven of these launches, the first of them
// over few, long rows, and its drain is what the chain fills: 60k-determinant 30-orbital space
// 429 us launched one after another, 336 chained; 64 spinors, M = 500k 8.85 -> 8.66 ms; full CI
// of 10 orbitals with 4 + 2 electrons, three vectors 117 -> 71 us.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// at the start of a chained kernel, launched with one CTA more than it has work for: true in
// that CTA, once the predecessor has completed
__device__ __forceinline__ bool chain_last_cta()
{
    chain_next();
    if (blockIdx.x != gridDim.x - 1) return false;
    chain_wait();
    return true;
}

template <typename... K, typename... A>
cudaError_t launch_chained(bool dependent, void (*kern)(K...), dim3 grid, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, (K)args...);
}

// ------------------------------------------------------------------ arithmetic policies
// The arithmetic of the bucket walks is a policy: staged element SC, table element TT,
// accumulator ACC, output TO, input coefficients CI; how a coefficient is read, multiplied
// in, renormalised (paired FP32) and written out.
template <typename TS, typename TC> struct PolF64 {   // FP64 / complex128
    static constexpr bool kFp64 = true;
    static constexpr bool kSplit = false;
    static constexpr bool kSkipSelf = true;
    using SC = TS;
    using TT = TS;
    using ACC = typename AccOf<TS>::type;
    using TO = ACC;
    using CI = TC;
    __device__ static SC load(const CI *C, int64_t i) { return (SC)C[i]; }
    __device__ static TT table(const TT *p) { return ldg(p); }
    __device__ static void clear(ACC &a) { zero(a); }
    __device__ static void mul_add(ACC &a, TT t, SC c) { fma_acc(a, t, c); }
    __device__ static void renorm(ACC &) {}
    __device__ static TO value(const ACC &a) { return a; }
    __device__ static void add_out(TO *p, TO v) { red_add(p, v); }
};
struct PolDS {   // paired FP32, real
    static constexpr bool kFp64 = false;
    static constexpr bool kSplit = true;
    static constexpr bool kSkipSelf = false;
    using SC = float2;
    using TT = float2;
    using ACC = Ds;
    using TO = double;
    using CI = float2;
    __device__ static SC load(const CI *C, int64_t i) { return C[i]; }
    __device__ static TT table(const TT *p) { return __ldg(p); }
    __device__ static void clear(ACC &a) { ds_zero(a); }
    __device__ static void mul_add(ACC &a, TT t, SC c) { ds_fma(a, t, c); }
    __device__ static void renorm(ACC &a) { ds_renorm(a); }
    __device__ static TO value(const ACC &a) { return ds_value(a); }
    __device__ static void add_out(TO *p, TO v) { red_add(p, v); }
};
struct PolF32 {   // FP32 storage, paired-FP32 sums
    static constexpr bool kFp64 = false;
    static constexpr bool kSplit = false;
    static constexpr bool kSkipSelf = false;
    using SC = float;
    using TT = float;
    using ACC = Ds;
    using TO = double;
    using CI = float;
    __device__ static SC load(const CI *C, int64_t i) { return C[i]; }
    __device__ static TT table(const TT *p) { return __ldg(p); }
    __device__ static void clear(ACC &a) { ds_zero(a); }
    __device__ static void mul_add(ACC &a, TT t, SC c);
    __device__ static void renorm(ACC &a) { ds_renorm(a); }
    __device__ static TO value(const ACC &a) { return ds_value(a); }
    __device__ static void add_out(TO *p, TO v) { red_add_nz(p, v); }
};
__device__ __forceinline__ void PolF32::mul_add(Ds &a, float t, float c) { ds_fma1(a, t, c); }
struct DsZ {
    Ds r, i;
};
struct PolDSZ {   // paired FP32, complex
    static constexpr bool kFp64 = false;
    static constexpr bool kSplit = true;
    static constexpr bool kSkipSelf = true;
    using SC = float4;
    using TT = float4;
    using ACC = DsZ;
    using TO = zdbl;
    using CI = float4;
    __device__ static SC load(const CI *C, int64_t i) { return C[i]; }
    __device__ static TT table(const TT *p) { return __ldg(p); }
    __device__ static void clear(ACC &a) { ds_zero(a.r), ds_zero(a.i); }
    __device__ static void mul_add(ACC &a, TT t, SC c)
    {
        const float2 tr_ = make_float2(t.x, t.y), ti = make_float2(t.z, t.w), mti = make_float2(-t.z, -t.w);
        const float2 cr = make_float2(c.x, c.y), ci = make_float2(c.z, c.w);
        ds_fma(a.r, tr_, cr);
        ds_fma(a.r, mti, ci);
        ds_fma(a.i, tr_, ci);
        ds_fma(a.i, ti, cr);
    }
    __device__ static void renorm(ACC &a) { ds_renorm(a.r), ds_renorm(a.i); }
    __device__ static TO value(const ACC &a) { return zdbl{ds_value(a.r), ds_value(a.i)}; }
    __device__ static void add_out(TO *p, TO v) { red_add(p, v); }
};

// ------------------------------------------------------------------ rules by policy and width
// the FP32-storage launch at 8 vectors
template <class P, int NV> constexpr bool f32_wide() { return NV >= 8 && sizeof(typename P::SC) == sizeof(float); }

// CTAs per SM that the bucket walks are held to: the gathers' latency asks for warps, the
// accumulators of a wide vector group for registers.  (Left to itself the compiler takes 40
// registers for one FP64 vector, 6 CTAs per SM.)
template <class P, int NV> constexpr int min_ctas()
{
    constexpr size_t b = NV * sizeof(typename P::SC);
    return f32_wide<P, NV>() ? SCI_F32_MINB : b <= 8 ? 8 : b <= 16 ? 6 : b <= 32 ? 5 : 4;
}
// ... and those of the aligned walk above kSortBucket members, whose threads walk hundreds of
// members: more registers let it hold more table loads in flight (60k-determinant 30-orbital
// space, one FP64 vector: 443 us at 8 CTAs, 227 at 6; 27 orbitals, two paired-FP32 vectors:
// 278 us at 6, 155 at 5; FP32 storage at 8 vectors loses, 596 us at 5, 617 at 4)
template <class P, int NV> constexpr int wide_ctas()
{
    constexpr int c = min_ctas<P, NV>();
    return f32_wide<P, NV>() ? c : c == 8 ? 6 : c == 6 ? 5 : c;
}
// Window rows of that walk: `rows` or 512 when they give kWindowsWanted windows, 16 an SM, three
// to four for each of its 4 to 6 resident CTAs, else 256 (a measured line: 60k space: 85 windows of 768 rows 227 us, 254 of 256 rows 148
// us; 40 orbitals, two vectors: 1,188 of 768 rows 1.21 ms, 3,563 of 256 1.14 ms; with 6,645
// windows of 768 rows, on the 2M space, 256 rows cost 3%).
constexpr int64_t kWindowsWanted = sci::kSMs * 16;
inline int window_rows(int64_t entries, int rows)
{
    for (int r : {rows, 512})
        if (r <= rows && entries / r >= kWindowsWanted) return r;
    return 256;
}
// The smallest bucket of the sorted kernel.  It pays where the products bind: FP64 at two and
// more vectors or complex (64 spinors, M = 500k, 5 to 64 members: 2.15 ms aligned, 1.41 ms
// sorted; 40 orbitals, two vectors: 0.83, 0.74; 30 orbitals at M = 500k, four vectors, whole
// kernel: 2.84, 2.60; whole products of 8 vectors, aligned up to 32 members against sorted: M =
// 400k 4.76, 4.58; M = 60k 1.87, 1.86; 14 orbitals 0.76, 0.69).  One FP64 vector is bound by the table gathers too, and the sort
// scatters a bucket's rows over warps: 33 to 64 members gain on the 60k space (206 -> 165 us)
// and lose little on the 2M one (2.78 -> 2.85 ms), smaller ones lose (2M: 3.48 ms from 5 on).
// The paired-FP32 sums (27 orbitals, one vector: 216 us aligned, 279 sorted; FP32 storage at
// 4 vectors and fewer) keep the aligned walk.  FP32 storage at 8 vectors, bound by
// instruction issue, sorts all buckets (30 orbitals, M = 500k: 2.48 ms aligned, 2.37 sorted,
// 2.44 with the register kernel's eight lanes per small bucket).
// A pair table of kSmallTable bytes or less stays close to the SMs, and one FP64 vector then
// sorts from 5 members on too (full CI of 10 orbitals, 0.1 MB: 245 us aligned, 228 sorted; 12
// orbitals, M = 20k, 0.24 MB: 63, 56).  Above it the aligned walk is the faster one again (M = 60k:
// 14 orbitals, 0.37 MB 142, 145; 16, 0.64 MB 110, 121; 18, 0.97 MB 101, 108).
constexpr int64_t kSmallTable = 1 << 18;
template <class P, int NV> constexpr int sort_from(bool small_table)
{
    if (f32_wide<P, NV>()) return 2;
    if (!P::kFp64) return kSortBucket + 1;
    return NV == 1 && sizeof(typename P::SC) == sizeof(double) && !small_table ? 33 : kSmallBucket + 1;
}
// Table entries up to which the paired-FP32 and FP32-storage launches take the buckets of at most
// kSortBucket members in the aligned walk of the larger ones instead of by size: a launch costs
// about 2 us, and these policies gain less by size than FP64 does.  Two paired-FP32 vectors, the
// product: 30 orbitals, 1,000 determinants (76k entries) 70 us by size, 43 in one walk; 3,000 (118k)
// 75, 45; full CI of 8 orbitals (137k) 51, 45; 40 orbitals, M = 60k, one vector (1.4M) 209, 228; FP32
// storage at 8 vectors, 221k entries 51, 60; 100 orbitals, 360k entries most of them in tiles, the
// deterministic mode at three vectors 2.25 ms, 2.41.
constexpr int64_t kFewEntries = 200'000;
// ... and in a row range in FP32 storage, when the space has larger buckets too, by the entries
// left to them: a short range owns few of a bucket's rows, and the launches by size stage and sort
// the others all the same.
// M = 400k, a 64th of the rows, 8 vectors (1.4M entries): 153 us by size, 140; M = 60k, an eighth,
// one vector (2.5M): 91, 84; M = 400k, an eighth, one vector (6.5M): 143, 162.  (Without larger
// buckets the windows are too short for the rows they own: full CI of 10 orbitals, a 64th, 8
// vectors, 221k entries: 51, 60.)
constexpr int64_t kFewRangeEntries = 3'000'000;
// b: the end of the tiles, large: of the buckets above kSortBucket members
template <class P, bool RANGED> constexpr bool in_one_walk(int64_t entries, int64_t b, int64_t large)
{
    if (P::kFp64) return false;
    return entries <= kFewEntries || (RANGED && !P::kSplit && large > b && entries - large <= kFewRangeEntries);
}
// The tiled walk takes 32 columns at a time as a mask of doubles for complex FP64 (64
// spinors, M = 500k: 1.43 -> 1.25 ms) and one FP64 vector (70 orbitals, M = 120k: doubles
// 1.25 -> 1.02 ms); otherwise in aligned groups (40 orbitals, two vectors: 1.22 ms, 1.29 by
// mask).
template <class P, int NV> __host__ __device__ constexpr bool mask_walk()
{
    return P::kFp64 && (NV == 1 || sizeof(typename P::SC) == sizeof(zdbl));
}

// where a launch over the vectors [v0, v0 + NV) finds coefficient v0 + v of determinant I: in
// C itself ([M][nvec]), or in the split copy of the vector group ([M][NV])
template <class P, int NV> __device__ __forceinline__ int64_t coef(int64_t I, int nvec, int v0, int v)
{
    return P::kSplit ? I * NV + v : I * nvec + v0 + v;
}

// ------------------------------------------------------------------ walking a row's doubles
// acc += sum over the set bits u of m of H(row, u) c_u: the pair-table loads of four members
// are issued before their products, and a member that is no double costs nothing.
template <class P, int NV>
__device__ __forceinline__ void walk_mask(uint32_t m, const typename P::TT *__restrict__ trow, const uint32_t *col,
                                          const typename P::SC *c, typename P::ACC (&acc)[NV])
{
    int n = __popc(m);
    for (; n >= kUnroll; n -= kUnroll) {
        int j[kUnroll];
        typename P::TT t[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; u++) {
            j[u] = __ffs((int)m) - 1;
            m &= m - 1;
            t[u] = P::table(trow + col[j[u]]);
        }
#pragma unroll
        for (int u = 0; u < kUnroll; u++)
#pragma unroll
            for (int v = 0; v < NV; v++) P::mul_add(acc[v], t[u], c[j[u] * NV + v]);
#pragma unroll
        for (int v = 0; v < NV; v++) P::renorm(acc[v]);
    }
    // one to three members left
    const bool two = n & 2, one = n & 1;
    int j0 = 0, j1 = 0, j2 = 0;
    typename P::TT t0{}, t1{}, t2{};
    if (two) {
        j0 = __ffs((int)m) - 1;
        m &= m - 1;
        j1 = __ffs((int)m) - 1;
        m &= m - 1;
        t0 = P::table(trow + col[j0]);
        t1 = P::table(trow + col[j1]);
    }
    if (one) {
        j2 = __ffs((int)m) - 1;
        t2 = P::table(trow + col[j2]);
    }
    if (two) {
#pragma unroll
        for (int v = 0; v < NV; v++) {
            P::mul_add(acc[v], t0, c[j0 * NV + v]);
            P::mul_add(acc[v], t1, c[j1 * NV + v]);
        }
    }
    if (one) {
#pragma unroll
        for (int v = 0; v < NV; v++) P::mul_add(acc[v], t2, c[j2 * NV + v]);
    }
#pragma unroll
    for (int v = 0; v < NV; v++) P::renorm(acc[v]);
}

// ------------------------------------------------------------------ doubles, small buckets
// Buckets of at most kSortBucket members.  A CTA owns the whole buckets that start in its
// kSortRows table rows, and works in three phases:
//   1. stage the members' codes, determinants and table columns;
//   2. each thread finds the doubles of its rows as a 64-bit mask over the bucket, gathers
//      the coefficients of the members that have any, and the CTA sorts the rows by their
//      number of doubles (a stable counting sort: neighbouring rows of a bucket stay
//      neighbours and share table sectors).  Rows without a double (27% of the entries of
//      the 2M-determinant 30-orbital space) end here;
//   3. each thread walks the set bits of a row's mask.  The rows of a warp have (nearly)
//      the same count, so its lanes stay on useful products: 97% of the FP64 lane slots
//      against 65% when lanes walk all members of their buckets.
constexpr int kSortRows = 448;
constexpr int kSortCap = kSortRows + kSortBucket;   // rows of a window, at most
constexpr int kSortRounds = kSortCap / kThreads;    // rows per thread in phases 1 and 2
static_assert(kSortCap % kThreads == 0, "phase 2 gives every thread the same number of rows");

template <class P, int NV> constexpr size_t sort_smem()
{
    return (size_t)kSortCap * (NV * sizeof(typename P::SC) + sizeof(uint2) + 4 * sizeof(uint32_t));
}

template <class P, int NV, bool RANGED, bool STORE>
__global__ void __launch_bounds__(kThreads, (min_ctas<P, NV>()))
k_doubles_sorted(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code,
                 const uint32_t *__restrict__ e_pos, int64_t E, sci::TabRule tr,
                 const typename P::TT *__restrict__ tab, const typename P::CI *__restrict__ C, int nvec, int v0, typename P::TO *__restrict__ Sout, sci::RowRange rr,
                 const uint32_t *__restrict__ slot)
{
    using SC = typename P::SC;
    constexpr int kWarps = kThreads / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint16_t s_hist[kWarps][64];
    __shared__ int s_base[64], s_total;
    if (chain_last_cta()) return;
    int64_t r0, r1;
    window(e_pos, E, kSortRows, r0, r1);
    if (r0 >= r1) return;
    const int W = (int)(r1 - r0);
    SC *s_c = reinterpret_cast<SC *>(smem);
    uint2 *s_mask = reinterpret_cast<uint2 *>(s_c + kSortCap * NV);
    uint32_t *s_code = reinterpret_cast<uint32_t *>(s_mask + kSortCap);
    uint32_t *s_col = s_code + kSortCap;
    uint32_t *s_idx = s_col + kSortCap;    // determinant, and the member's parity in bit 31
    uint32_t *s_row = s_idx + kSortCap;    // sorted rows: window row | start of its bucket << 16
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // warp w holds the rows [w * per, (w + 1) * per), 32 at a time
    const int per = ((W + kWarps - 1) / kWarps + 31) & ~31;

    uint32_t pos[kSortRounds];
#pragma unroll
    for (int k = 0; k < kSortRounds; k++) {
        const int q = wid * per + 32 * k + lane;
        pos[k] = 0;
        if (32 * k < per && q < W) {
            const uint32_t code = e_code[r0 + q];
            pos[k] = e_pos[r0 + q];
            uint32_t rowoff, colbase;
            sci::pair_offsets(tr, sci::code_x(code), sci::code_y(code), rowoff, colbase);
            s_code[q] = col_code(code);
            s_col[q] = colbase;
            s_idx[q] = e_idx[r0 + q] | (uint32_t)sci::code_par(code) << 31;
        }
    }
    for (int t = threadIdx.x; t < kWarps * 64; t += kThreads) (&s_hist[0][0])[t] = 0;
    __syncthreads();

    int key[kSortRounds], rank[kSortRounds];
#pragma unroll
    for (int k = 0; k < kSortRounds; k++) {
        const int q = wid * per + 32 * k + lane;
        key[k] = -1;
        if (pos[k] != 0) {
            const int size = sci::pos_size(pos[k]), bs = q - sci::pos_off(pos[k]);
            const uint32_t cc = s_code[q];
            const uint32_t rc = __byte_perm(cc, 0, 0x1010);   // (x, y, x, y) of the row
            uint2 m = make_uint2(doubles_mask(rc, s_code + bs, min(size, 32)), 0u);
            if (size > 32) m.y = doubles_mask(rc, s_code + bs + 32, size - 32);
            s_mask[q] = m;
            const int deg = __popc(m.x) + __popc(m.y);
            const uint32_t ip = s_idx[q];
            const int64_t I = ip & 0x7fffffffu;
            if (deg) {
#pragma unroll
                for (int v = 0; v < NV; v++) s_c[q * NV + v] = flip(ip >> 31, P::load(C, coef<P, NV>(I, nvec, v0, v)));
                if (!RANGED || (I >= rr.rb && I < rr.re)) key[k] = 63 - deg;
            } else if constexpr (STORE) {   // the slot of a row without doubles holds a zero
#pragma unroll
                for (int v = 0; v < NV; v++) Sout[(int64_t)slot[r0 + q] * nvec + v0 + v] = typename P::TO{};
            }
        }
        rank[k] = sci::sort_rank(key[k], s_hist[wid], lane);
    }
    __syncthreads();
    if (wid == 0) sci::sort_prefix<kWarps>(s_hist, lane, s_base, s_total);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSortRounds; k++)
        if (key[k] >= 0) {
            const int q = wid * per + 32 * k + lane;
            s_row[s_base[key[k]] + s_hist[wid][key[k]] + rank[k]] =
                (uint32_t)q | (uint32_t)(q - sci::pos_off(pos[k])) << 16;
        }
    __syncthreads();

    const int nrows = s_total;
    for (int t = threadIdx.x; t < nrows; t += kThreads) {
        const uint32_t row = s_row[t];
        const int q = (int)(row & 0xFFFFu), bs = (int)(row >> 16);
        const uint32_t cc = s_code[q];
        uint32_t rowoff, colbase;
        sci::pair_offsets(tr, (int)(cc & 0xFFu), (int)((cc >> 8) & 0xFFu), rowoff, colbase);
        const typename P::TT *trow = tab + rowoff;
        const uint2 m = s_mask[q];
        typename P::ACC acc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) P::clear(acc[v]);
        walk_mask<P, NV>(m.x, trow, s_col + bs, s_c + bs * NV, acc);
        if (m.y) walk_mask<P, NV>(m.y, trow, s_col + bs + 32, s_c + (bs + 32) * NV, acc);
        const uint32_t ip = s_idx[q];
        const bool par = ip >> 31;
        if constexpr (STORE) {
#pragma unroll
            for (int v = 0; v < NV; v++) Sout[(int64_t)slot[r0 + q] * nvec + v0 + v] = flip(par, P::value(acc[v]));
        } else {
#pragma unroll
            for (int v = 0; v < NV; v++)
                P::add_out(Sout + (int64_t)(ip & 0x7fffffffu) * nvec + v0 + v, flip(par, P::value(acc[v])));
        }
    }
}

// ------------------------------------------------------------------ doubles, smallest buckets
// Buckets of S <= kSmallBucket members, which are most of the entries of a selected space
// (62% of the 2M-determinant 30-orbital space) but few of its pairs (7%).  NV lanes take a
// bucket, one vector each, with the members in registers: no staging, no barrier, and the
// members without a double read no coefficient and add nothing.  Lanes of one bucket read the
// same table entries and neighbouring coefficients.  The L1's rate of scattered 8-byte accesses
// bounds it (2M space: 145M entries in 0.79 ms); two or four buckets in flight per thread were
// slower (0.88 ms).
template <class P, int S, int NV, bool RANGED, bool STORE>
__global__ void __launch_bounds__(kThreads)
k_doubles_small(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code, int64_t nbuckets,
                sci::TabRule tr, const typename P::TT *__restrict__ tab, const typename P::CI *__restrict__ C,
                int nvec, int v0, typename P::TO *__restrict__ Sout, sci::RowRange rr,
                const uint32_t *__restrict__ slot)
{
    if (chain_last_cta()) return;
    const int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x;
    const int v = (int)(t % NV);
    const int64_t b = t / NV;
    if (b >= nbuckets) return;
    const int64_t g = b * S;
    uint32_t code[S];
#pragma unroll
    for (int i = 0; i < S; i++) code[i] = e_code[g + i];
    unsigned d[S];   // bit j of d[i]: members i and j are doubles of each other
#pragma unroll
    for (int i = 0; i < S; i++) d[i] = 0;
#pragma unroll
    for (int i = 0; i < S; i++)
#pragma unroll
        for (int j = i + 1; j < S; j++)
            if (disjoint(row_code(code[i]), col_code(code[j]))) d[i] |= 1u << j, d[j] |= 1u << i;
    unsigned any = 0;
#pragma unroll
    for (int i = 0; i < S; i++) any |= d[i];
    if (!STORE && any == 0) return;
    int64_t idx[S];
    typename P::SC c[S];
    uint32_t rowoff[S], colbase[S];
#pragma unroll
    for (int i = 0; i < S; i++) {
        idx[i] = 0;
        c[i] = typename P::SC{};
        if (d[i]) {
            idx[i] = e_idx[g + i];
            c[i] = flip(sci::code_par(code[i]), P::load(C, coef<P, NV>(idx[i], nvec, v0, v)));
        }
        sci::pair_offsets(tr, sci::code_x(code[i]), sci::code_y(code[i]), rowoff[i], colbase[i]);
    }
    typename P::TT h[S][S];
#pragma unroll
    for (int i = 0; i < S; i++)
#pragma unroll
        for (int j = 0; j < S; j++) {
            h[i][j] = typename P::TT{};
            if (i != j && (d[i] >> j & 1)) h[i][j] = P::table(tab + rowoff[i] + colbase[j]);
        }
#pragma unroll
    for (int i = 0; i < S; i++) {
        typename P::ACC acc;
        P::clear(acc);
#pragma unroll
        for (int j = 0; j < S; j++)
            if (i != j && (d[i] >> j & 1)) P::mul_add(acc, h[i][j], c[j]);
        P::renorm(acc);
        const typename P::TO out = flip(sci::code_par(code[i]), P::value(acc));
        if constexpr (STORE) {
            Sout[(int64_t)slot[g + i] * nvec + v0 + v] = out;
        } else if (d[i] && (!RANGED || (idx[i] >= rr.rb && idx[i] < rr.re))) {
            P::add_out(Sout + idx[i] * nvec + v0 + v, out);
        }
    }
}

// ------------------------------------------------------------------ doubles, aligned walk
// A CTA stages the whole buckets that start in its CH table rows, and each thread walks the
// members of its row's bucket in order, kUnroll at a time: lanes of one bucket read the same
// member and neighbouring table entries at every step.  A group with no double of the row is
// skipped; in the others a member that is no double adds t = 0.
template <class P, int NV, bool RANGED, bool STORE, int MINB>
__global__ void __launch_bounds__(kThreads, MINB)
k_doubles_aligned(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code,
                  const uint32_t *__restrict__ e_pos, int64_t E, int CH, sci::TabRule tr,
                  const typename P::TT *__restrict__ tab, const typename P::CI *__restrict__ C, int nvec, int v0, typename P::TO *__restrict__ Sout, sci::RowRange rr,
                  const uint32_t *__restrict__ slot)
{
    using SC = typename P::SC;
    using TT = typename P::TT;
    extern __shared__ __align__(16) unsigned char smem[];
    if (chain_last_cta()) return;
    int64_t r0, r1;
    window(e_pos, E, CH, r0, r1);
    if (r0 >= r1) return;
    const int W = (int)(r1 - r0);
    SC *s_c = reinterpret_cast<SC *>(smem);
    const size_t cbytes = ((size_t)W * NV * sizeof(SC) + 15) & ~(size_t)15;
    uint2 *s_kc = reinterpret_cast<uint2 *>(smem + cbytes);
    uint16_t *s_own = reinterpret_cast<uint16_t *>(smem + cbytes + (size_t)W * sizeof(uint2));
    int nrows = W;
    if constexpr (RANGED) {
        nrows = owned_rows(e_idx, r0, W, rr, s_own);
        if (nrows == 0) return;
    }
    for (int q = threadIdx.x; q < W; q += blockDim.x) {
        const int64_t g = r0 + q;
        const uint32_t idx = e_idx[g], code = e_code[g];
        uint32_t rowoff, colbase;
        sci::pair_offsets(tr, sci::code_x(code), sci::code_y(code), rowoff, colbase);
        s_kc[q] = make_uint2(col_code(code), colbase);
        const bool par = sci::code_par(code);
#pragma unroll
        for (int v = 0; v < NV; v++) s_c[q * NV + v] = flip(par, P::load(C, coef<P, NV>(idx, nvec, v0, v)));
    }
    __syncthreads();
    for (int t_ = threadIdx.x; t_ < nrows; t_ += blockDim.x) {
        const int q0 = RANGED ? (int)s_own[t_] : t_;
        const uint32_t code = e_code[r0 + q0], pos = e_pos[r0 + q0];
        uint32_t rowoff, colbase;
        sci::pair_offsets(tr, sci::code_x(code), sci::code_y(code), rowoff, colbase);
        // FP64 policies walk the members other than the row itself, j standing for bucket
        // position j + (j >= q0); the paired-FP32 ones all members (see the policies)
        const int bs = q0 - sci::pos_off(pos), je = bs + sci::pos_size(pos) - (P::kSkipSelf ? 1 : 0);
        auto member = [&](int j) { return P::kSkipSelf ? j + (j >= q0) : j; };
        const uint32_t rc = row_code(code);
        const TT *trow = tab + rowoff;
        typename P::ACC acc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) P::clear(acc[v]);
        int j = bs;
        for (; j + kUnroll <= je; j += kUnroll) {
            uint2 kc[kUnroll];
            TT t[kUnroll];
            unsigned vm = 0;
#pragma unroll
            for (int u = 0; u < kUnroll; u++) {
                kc[u] = s_kc[member(j + u)];
                vm |= (unsigned)disjoint(rc, kc[u].x) << u;
            }
            if (vm == 0) continue;
#pragma unroll
            for (int u = 0; u < kUnroll; u++) {
                t[u] = TT{};
                if (vm & (1u << u)) t[u] = P::table(trow + kc[u].y);
            }
#pragma unroll
            for (int u = 0; u < kUnroll; u++)
#pragma unroll
                for (int v = 0; v < NV; v++) P::mul_add(acc[v], t[u], s_c[member(j + u) * NV + v]);
#pragma unroll
            for (int v = 0; v < NV; v++) P::renorm(acc[v]);
        }
        for (; j < je; j++) {
            const int m = member(j);
            const uint2 kc = s_kc[m];
            if (!disjoint(rc, kc.x)) continue;
            const TT t = P::table(trow + kc.y);
#pragma unroll
            for (int v = 0; v < NV; v++) P::mul_add(acc[v], t, s_c[m * NV + v]);
        }
        const bool par = sci::code_par(code);
        if constexpr (STORE) {
#pragma unroll
            for (int v = 0; v < NV; v++) Sout[(int64_t)slot[r0 + q0] * nvec + v0 + v] = flip(par, P::value(acc[v]));
        } else {
            const uint32_t idx = e_idx[r0 + q0];
#pragma unroll
            for (int v = 0; v < NV; v++) P::add_out(Sout + (int64_t)idx * nvec + v0 + v, flip(par, P::value(acc[v])));
        }
    }
}

// ------------------------------------------------------------------ doubles, tiled
// (N-2) buckets of more than tile_b members (sci_set_tile_threshold) are too large to
// stage whole beside a window, so they run here.  A CTA takes kTileRows consecutive
// members of one bucket as its rows (one per thread) and streams the bucket's members
// through shared memory in column tiles, each staged once per CTA; every thread walks a
// column tile against its row as the window kernels walk a bucket (disjointness test, one
// table load per double, the FMAs), so a row sums the same products.  The row itself and
// its single excitations fail the disjointness test and add nothing.  All threads of a
// CTA share the bucket, so trip counts are uniform and the barriers are CTA-wide.
// shared memory of the tiled kernel: at most this, which needs no opt-in
constexpr size_t kTiledSmem = 48 * 1024;

// C holds coefficient v of determinant I at C[coef<P, NV>(I, nvec, v0, v)].  With few tiles
// (a handful of very large buckets) the columns of a bucket are also split: CTA row y of
// the grid (gridDim.y = nsplit) takes the y-th of nsplit equal runs of column tiles and
// adds its partial row sums atomically (nsplit = 1 in the deterministic mode, where one
// CTA writes a slot).
template <class P, int NV, bool RANGED, bool STORE>
__global__ void __launch_bounds__(kThreads)
k_doubles_tiled(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code,
                const uint32_t *__restrict__ e_pos, const uint32_t *__restrict__ tiles, int64_t ntiles, int TCOL,
                sci::TabRule tr, const typename P::TT *__restrict__ tab, const typename P::CI *__restrict__ C,
                int nvec, int v0, typename P::TO *__restrict__ Sout, sci::RowRange rr,
                const uint32_t *__restrict__ slot)
{
    if (chain_last_cta()) return;
    const int nsplit = STORE ? 1 : (int)gridDim.y;
    using SC = typename P::SC;
    using TT = typename P::TT;
    using ACC = typename P::ACC;
    extern __shared__ __align__(16) unsigned char smem[];
    SC *s_c = reinterpret_cast<SC *>(smem);
    // codes and columns, apart for the walk by masks and as pairs for the aligned one
    uint32_t *s_code = reinterpret_cast<uint32_t *>(smem + (((size_t)TCOL * NV * sizeof(SC) + 15) & ~(size_t)15));
    uint32_t *s_col = s_code + TCOL;
    uint2 *s_kc = reinterpret_cast<uint2 *>(s_code);
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x - 1) {
        const int64_t r0 = tiles[t];
        const uint32_t pos0 = e_pos[r0];
        const int64_t bs = r0 - sci::pos_off(pos0);
        const int bsize = sci::pos_size(pos0);
        // this CTA's column tiles: [c_lo, c_hi) in members of the bucket
        const int nct = (bsize + TCOL - 1) / TCOL, per_split = (nct + nsplit - 1) / nsplit;
        const int c_lo = (int)blockIdx.y * per_split * TCOL, c_hi = min(bsize, c_lo + per_split * TCOL);
        if (c_lo >= c_hi) continue;   // uniform over the CTA
        const int64_t row = r0 + threadIdx.x;
        bool active = row < bs + bsize;
        if (RANGED && active) {
            const int64_t I = e_idx[row];
            active = I >= rr.rb && I < rr.re;
        }
        if (!__syncthreads_or(active)) continue;   // no row of this tile is computed
        uint32_t rc = 0;
        const TT *trow = tab;
        bool par = false;
        if (active) {
            const uint32_t code = e_code[row];
            uint32_t rowoff, colbase;
            sci::pair_offsets(tr, sci::code_x(code), sci::code_y(code), rowoff, colbase);
            rc = row_code(code);
            trow = tab + rowoff;
            par = sci::code_par(code);
        }
        ACC acc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) P::clear(acc[v]);
        for (int cs = c_lo; cs < c_hi; cs += TCOL) {
            const int n = min(TCOL, c_hi - cs);
            __syncthreads();   // every thread is done with the previous column tile
            for (int q = threadIdx.x; q < n; q += blockDim.x) {
                const int64_t g = bs + cs + q;
                const uint32_t idx = e_idx[g], code = e_code[g];
                uint32_t rowoff, colbase;
                sci::pair_offsets(tr, sci::code_x(code), sci::code_y(code), rowoff, colbase);
                if constexpr (mask_walk<P, NV>()) {
                    s_code[q] = col_code(code);
                    s_col[q] = colbase;
                } else {
                    s_kc[q] = make_uint2(col_code(code), colbase);
                }
                const bool pq = sci::code_par(code);
#pragma unroll
                for (int v = 0; v < NV; v++) s_c[q * NV + v] = flip(pq, P::load(C, coef<P, NV>(idx, nvec, v0, v)));
            }
            __syncthreads();
            if (!active) continue;
            if constexpr (mask_walk<P, NV>()) {
                for (int j = 0; j < n; j += 32)
                    walk_mask<P, NV>(doubles_mask(rc, s_code + j, min(32, n - j)), trow, s_col + j, s_c + j * NV, acc);
            } else {
                int j = 0;
                for (; j + kUnroll <= n; j += kUnroll) {
                    uint2 kc[kUnroll];
                    TT tv[kUnroll];
                    unsigned vm = 0;
#pragma unroll
                    for (int u = 0; u < kUnroll; u++) {
                        kc[u] = s_kc[j + u];
                        vm |= (unsigned)disjoint(rc, kc[u].x) << u;
                    }
                    if (vm == 0) continue;
#pragma unroll
                    for (int u = 0; u < kUnroll; u++) {
                        tv[u] = TT{};
                        if (vm & (1u << u)) tv[u] = P::table(trow + kc[u].y);
                    }
#pragma unroll
                    for (int u = 0; u < kUnroll; u++)
#pragma unroll
                        for (int v = 0; v < NV; v++) P::mul_add(acc[v], tv[u], s_c[(j + u) * NV + v]);
#pragma unroll
                    for (int v = 0; v < NV; v++) P::renorm(acc[v]);
                }
                for (; j < n; j++) {
                    const uint2 kc = s_kc[j];
                    if (!disjoint(rc, kc.x)) continue;
                    const TT tv = P::table(trow + kc.y);
#pragma unroll
                    for (int v = 0; v < NV; v++) P::mul_add(acc[v], tv, s_c[j * NV + v]);
                }
#pragma unroll
                for (int v = 0; v < NV; v++) P::renorm(acc[v]);
            }
        }
        if (active) {
            if constexpr (STORE) {
#pragma unroll
                for (int v = 0; v < NV; v++) Sout[(int64_t)slot[row] * nvec + v0 + v] = flip(par, P::value(acc[v]));
            } else {
                const uint32_t idx = e_idx[row];
#pragma unroll
                for (int v = 0; v < NV; v++) P::add_out(Sout + (int64_t)idx * nvec + v0 + v, flip(par, P::value(acc[v])));
            }
        }
    }
}

// ------------------------------------------------------------------ singles
template <typename TS, typename TC, int NV, bool RANGED, bool STORE = false, int KW = 1>
__global__ void __launch_bounds__(kThreads)
k_singles(const uint32_t *__restrict__ e_idx, const uint64_t *__restrict__ e_S, const uint32_t *__restrict__ e_meta,
          int64_t E, int norb, sci::RefW ref, const TS *__restrict__ fref, const TS *__restrict__ g_so,
          const TC *__restrict__ C, int nvec, int v0, typename AccOf<TS>::type *__restrict__ Sout, sci::RowRange rr, const uint32_t *__restrict__ slot)
{
    using TA = typename AccOf<TS>::type;
    chain_next();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x) {
        if constexpr (RANGED) {
            const int64_t I = e_idx[p];
            if (I < rr.rb || I >= rr.re) continue;
        }
        const uint32_t meta = e_meta[p];
        const int a = sci::meta_x(meta);
        const bool par = sci::meta_par(meta);
        const int64_t bs = p - (int64_t)sci::meta_off(meta);
        const int64_t be = bs + (int64_t)sci::meta_size(meta);
        uint64_t part[KW], holes[KW];   // S \ ref and ref \ S, word w holding orbitals 64w..64w+63
#pragma unroll
        for (int w_ = 0; w_ < KW; w_++) {
            const uint64_t Sw = e_S[p * KW + w_], rw = ref.w[w_];
            part[w_] = Sw & ~rw, holes[w_] = rw & ~Sw;
        }
        TA acc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) zero(acc[v]);
        for (int64_t q = bs; q < be; q++) {
            if (q == p) continue;
            const uint32_t mq = e_meta[q];
            const int i = sci::meta_x(mq);
            const bool parq = sci::meta_par(mq);
            const uint32_t idxq = e_idx[q];
            TS f = ldg(fref + i * norb + a);
#pragma unroll
            for (int w_ = 0; w_ < KW; w_++)
            for (uint64_t m = part[w_]; m; m &= m - 1) {
                int k = 64 * w_ + __ffsll((long long)m) - 1;
                TS g = ldg(g_so + ((int64_t)k * norb + i) * norb + a);
                if constexpr (sizeof(TS) == sizeof(zdbl)) { f.x += g.x; f.y += g.y; } else { f += g; }
            }
#pragma unroll
            for (int w_ = 0; w_ < KW; w_++)
            for (uint64_t m = holes[w_]; m; m &= m - 1) {
                int k = 64 * w_ + __ffsll((long long)m) - 1;
                TS g = ldg(g_so + ((int64_t)k * norb + i) * norb + a);
                if constexpr (sizeof(TS) == sizeof(zdbl)) { f.x -= g.x; f.y -= g.y; } else { f -= g; }
            }
#pragma unroll
            for (int v = 0; v < NV; v++) fma_acc(acc[v], f, flip(parq, C[(int64_t)idxq * nvec + v0 + v]));
        }
        if constexpr (STORE) {
#pragma unroll
            for (int v = 0; v < NV; v++) Sout[(int64_t)slot[p] * nvec + v0 + v] = flip(par, acc[v]);
        } else {
            const uint32_t idx = e_idx[p];
#pragma unroll
            for (int v = 0; v < NV; v++) red_add(Sout + (int64_t)idx * nvec + v0 + v, flip(par, acc[v]));
        }
    }
    chain_wait();
}

// ------------------------------------------------------------------ singles, paired FP32
// F^S_ai = F^ref_ai + sum_{k in S\ref} g_ai(k) - sum_{k in ref\S} g_ai(k) summed in
// paired FP32 from split copies of fref and g_so, then multiplied into the row sum like
// the doubles.  C2/C4 is the split vector group (row stride NV).
using sci::ds_add;

template <int NV, bool RANGED, bool STORE = false, int KW = 1>
__global__ void __launch_bounds__(kThreads)
k_singles_ds(const uint32_t *__restrict__ e_idx, const uint64_t *__restrict__ e_S, const uint32_t *__restrict__ e_meta,
             int64_t E, int norb, sci::RefW ref, const float2 *__restrict__ fref2, const float2 *__restrict__ g2,
             const float2 *__restrict__ C2, int nvec, int v0, double *__restrict__ Sout, sci::RowRange rr, const uint32_t *__restrict__ slot)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x) {
        if constexpr (RANGED) {
            const int64_t I = e_idx[p];
            if (I < rr.rb || I >= rr.re) continue;
        }
        const uint32_t meta = e_meta[p];
        const int a = sci::meta_x(meta);
        const bool par = sci::meta_par(meta);
        const int64_t bs = p - (int64_t)sci::meta_off(meta);
        const int64_t be = bs + (int64_t)sci::meta_size(meta);
        uint64_t part[KW], holes[KW];   // S \ ref and ref \ S, word w holding orbitals 64w..64w+63
#pragma unroll
        for (int w_ = 0; w_ < KW; w_++) {
            const uint64_t Sw = e_S[p * KW + w_], rw = ref.w[w_];
            part[w_] = Sw & ~rw, holes[w_] = rw & ~Sw;
        }
        Ds acc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) ds_zero(acc[v]);
        for (int64_t q = bs; q < be; q++) {
            if (q == p) continue;
            const uint32_t mq = e_meta[q];
            const int i = sci::meta_x(mq);
            const bool parq = sci::meta_par(mq);
            const uint32_t idxq = e_idx[q];
            const float2 f0 = __ldg(fref2 + i * norb + a);
            Ds f{f0.x, f0.y};
#pragma unroll
            for (int w_ = 0; w_ < KW; w_++)
            for (uint64_t m = part[w_]; m; m &= m - 1) {
                const int k = 64 * w_ + __ffsll((long long)m) - 1;
                ds_add(f, __ldg(g2 + ((int64_t)k * norb + i) * norb + a));
            }
#pragma unroll
            for (int w_ = 0; w_ < KW; w_++)
            for (uint64_t m = holes[w_]; m; m &= m - 1) {
                const int k = 64 * w_ + __ffsll((long long)m) - 1;
                ds_add(f, flip(true, __ldg(g2 + ((int64_t)k * norb + i) * norb + a)));
            }
            ds_renorm(f);
            const float2 fv = make_float2(f.hi, f.lo);
#pragma unroll
            for (int v = 0; v < NV; v++) ds_fma(acc[v], fv, flip(parq, C2[(int64_t)idxq * NV + v]));
        }
        if constexpr (STORE) {
#pragma unroll
            for (int v = 0; v < NV; v++) Sout[(int64_t)slot[p] * nvec + v0 + v] = flip(par, ds_value(acc[v]));
        } else {
            const uint32_t idx = e_idx[p];
#pragma unroll
            for (int v = 0; v < NV; v++) red_add(Sout + (int64_t)idx * nvec + v0 + v, flip(par, ds_value(acc[v])));
        }
    }
}

template <int NV, bool RANGED, bool STORE = false, int KW = 1>
__global__ void __launch_bounds__(kThreads)
k_singles_dsz(const uint32_t *__restrict__ e_idx, const uint64_t *__restrict__ e_S,
              const uint32_t *__restrict__ e_meta, int64_t E, int norb, sci::RefW ref,
              const float4 *__restrict__ fref4, const float4 *__restrict__ g4, const float4 *__restrict__ C4,
              int nvec, int v0, zdbl *__restrict__ Sout, sci::RowRange rr, const uint32_t *__restrict__ slot)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x) {
        if constexpr (RANGED) {
            const int64_t I = e_idx[p];
            if (I < rr.rb || I >= rr.re) continue;
        }
        const uint32_t meta = e_meta[p];
        const int a = sci::meta_x(meta);
        const bool par = sci::meta_par(meta);
        const int64_t bs = p - (int64_t)sci::meta_off(meta);
        const int64_t be = bs + (int64_t)sci::meta_size(meta);
        uint64_t part[KW], holes[KW];   // S \ ref and ref \ S, word w holding orbitals 64w..64w+63
#pragma unroll
        for (int w_ = 0; w_ < KW; w_++) {
            const uint64_t Sw = e_S[p * KW + w_], rw = ref.w[w_];
            part[w_] = Sw & ~rw, holes[w_] = rw & ~Sw;
        }
        Ds ar[NV], ai[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) ds_zero(ar[v]), ds_zero(ai[v]);
        for (int64_t q = bs; q < be; q++) {
            if (q == p) continue;
            const uint32_t mq = e_meta[q];
            const int i = sci::meta_x(mq);
            const bool parq = sci::meta_par(mq);
            const uint32_t idxq = e_idx[q];
            const float4 f0 = __ldg(fref4 + i * norb + a);
            Ds fr{f0.x, f0.y}, fi{f0.z, f0.w};
#pragma unroll
            for (int w_ = 0; w_ < KW; w_++)
            for (uint64_t m = part[w_]; m; m &= m - 1) {
                const int k = 64 * w_ + __ffsll((long long)m) - 1;
                const float4 g = __ldg(g4 + ((int64_t)k * norb + i) * norb + a);
                ds_add(fr, make_float2(g.x, g.y));
                ds_add(fi, make_float2(g.z, g.w));
            }
#pragma unroll
            for (int w_ = 0; w_ < KW; w_++)
            for (uint64_t m = holes[w_]; m; m &= m - 1) {
                const int k = 64 * w_ + __ffsll((long long)m) - 1;
                const float4 g = flip(true, __ldg(g4 + ((int64_t)k * norb + i) * norb + a));
                ds_add(fr, make_float2(g.x, g.y));
                ds_add(fi, make_float2(g.z, g.w));
            }
            ds_renorm(fr);
            ds_renorm(fi);
            const float2 tr_ = make_float2(fr.hi, fr.lo), ti = make_float2(fi.hi, fi.lo);
            const float2 mti = make_float2(-fi.hi, -fi.lo);
#pragma unroll
            for (int v = 0; v < NV; v++) {
                const float4 c = flip(parq, C4[(int64_t)idxq * NV + v]);
                const float2 cr = make_float2(c.x, c.y), ci = make_float2(c.z, c.w);
                ds_fma(ar[v], tr_, cr);
                ds_fma(ar[v], mti, ci);
                ds_fma(ai[v], tr_, ci);
                ds_fma(ai[v], ti, cr);
            }
        }
        if constexpr (STORE) {
#pragma unroll
            for (int v = 0; v < NV; v++) Sout[(int64_t)slot[p] * nvec + v0 + v] = flip(par, zdbl{ds_value(ar[v]), ds_value(ai[v])});
        } else {
            const uint32_t idx = e_idx[p];
#pragma unroll
            for (int v = 0; v < NV; v++)
                red_add(Sout + (int64_t)idx * nvec + v0 + v, flip(par, zdbl{ds_value(ar[v]), ds_value(ai[v])}));
        }
    }
}

int grid_for(int64_t n, int threads = kThreads)
{
    int64_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > sci::kSMs * 32) g = sci::kSMs * 32;
    return (int)g;
}

// Rows per CTA (CH) so that the staged window, at most CH + maxb - 1 members, fits the
// shared-memory budget; small windows first (more resident CTAs per SM), larger ones
// only when the buckets need them.
int choose_rows(int maxb, size_t bytes_per_entry, size_t &smem, int max_rows = kRowsPerCta)
{
    const size_t budgets[3] = {48 * 1024, 100 * 1024, 200 * 1024};
    for (size_t budget : budgets) {
        int64_t ch = (int64_t)(budget / bytes_per_entry) - (int64_t)maxb - 8;
        if (ch >= 512 || (budget == budgets[2] && ch >= 64)) {
            ch = std::min<int64_t>(ch, max_rows);
            ch = std::max<int64_t>(64, ch & ~(int64_t)63);
            smem = (size_t)(ch + maxb) * bytes_per_entry + 64;
            return (int)ch;
        }
    }
    return -1;
}

sci::TabRule tab_rule(const sci_ctx *ctx) { return sci::TabRule{ctx->spinors, ctx->n}; }

// The tables a sigma launch walks and the rows it computes: the full tables (every row),
// or the range tables of sci_set_row_range() (rows [row_b, row_e)).
// The (N-2) entries [0, sp.big) are the buckets of the tiled kernel (tile starts in
// tiles[0, sp.ntiles)); the window kernels walk [sp.big, e2), whose largest bucket is
// sp.maxb_small.  A launch takes the wide split when it stages kWideRowBytes or more per
// window row.
struct Tabs {
    const uint32_t *e2_idx, *e2_code, *e2_pos;
    int64_t e2;
    const uint32_t *e1_idx;
    const uint64_t *e1_S;
    const uint32_t *e1_meta;
    int64_t e1;
    sci::RowRange rr;
    const sci::TileSplit *ts;
    const uint32_t *tiles() const { return ts->tiles; }
    const sci::Split &split(size_t row_bytes) const
    {
        return row_bytes >= sci::kWideRowBytes ? ts->wide : ts->base;
    }
    int maxb_small() const { return ts->base.maxb_small; }   // the larger of the two
};

Tabs tabs_of(const sci_ctx *ctx)
{
    if (ctx->ranged)
        return Tabs{ctx->r2_idx, ctx->r2_code, ctx->r2_pos, ctx->r2, ctx->r1_idx, ctx->r1_S, ctx->r1_meta, ctx->r1,
                    sci::RowRange{ctx->row_b, ctx->row_e}, &ctx->rsplit2};
    return Tabs{ctx->e2_idx, ctx->e2_code, ctx->e2_pos, ctx->e2, ctx->e1_idx, ctx->e1_S, ctx->e1_meta, ctx->e1,
                sci::RowRange{0, ctx->M}, &ctx->split2};
}

// the tiled kernel over the buckets of [0, sp.big) (nothing when there are none)
template <class P, bool RG, bool ST, int NV>
int launch_tiled(sci_ctx *ctx, const Tabs &T, const sci::Split &sp, const typename P::TT *tab,
                 const typename P::CI *C, int nvec, int v0, typename P::TO *S, bool &chained)
{
    if (sp.ntiles == 0) return SCI_OK;
    const size_t per = NV * sizeof(typename P::SC) + sizeof(uint2);
    int tcol = (int)std::min<size_t>(1024, (kTiledSmem - 16) / per) & ~31;
    // with few tiles the columns are split too, in runs of 64 members and more, for four
    // waves of CTAs: tiles of unequal buckets leave the last wave nearly empty otherwise (not
    // in the deterministic mode, whose slots have one writer).  70 orbitals, M = 120k: 942 us
    // at one wave, 823 at four; 45 spinors, M = 118k, two paired-FP32 vectors: 234 tiles, 181
    // us unsplit, 121.  Wide vector groups pay for each split with as many atomics per row
    // and stop at one wave (56 orbitals, 8 vectors: 6.43 ms at one, 6.84 at four).
    int nsplit = 1;
    const int64_t ctas = sci::kSMs * (NV * sizeof(typename P::SC) >= sci::kWideRowBytes ? 8 : 32);
    if (!ST && sp.ntiles < ctas) {
        const int64_t want = (ctas + sp.ntiles - 1) / sp.ntiles;
        const int cols = (int)std::max<int64_t>(64, ((ctx->maxb2 + want - 1) / want + 31) & ~(int64_t)31);
        tcol = std::min(tcol, cols);
        nsplit = (int)std::min<int64_t>({want, (ctx->maxb2 + tcol - 1) / tcol, 65535});
    }
    const size_t smem = (((size_t)tcol * NV * sizeof(typename P::SC) + 15) & ~(size_t)15) + (size_t)tcol * sizeof(uint2);
    cudaError_t e = launch_chained(chained, k_doubles_tiled<P, NV, RG, ST>,
                                   dim3((unsigned)sp.ntiles + 1, (unsigned)nsplit), smem, ctx->stream, T.e2_idx,
                                   T.e2_code, T.e2_pos, T.tiles(), sp.ntiles, tcol, tab_rule(ctx), tab, C, nvec, v0, S,
                                   T.rr, ST ? ctx->det_inv2 : nullptr);
    chained = true;
    return sci_cuda_check(ctx, e, "k_doubles_tiled launch");
}

// staged bytes per window row: NV coefficients, the (code, offset) pair, and in a RANGED
// launch the row's slot in the owned-row list
template <bool RG> constexpr size_t row_extra() { return RG ? 8 + sizeof(uint16_t) : 8; }

// the doubles of one vector group, by bucket size: the tiled kernel above the tile threshold,
// the aligned walk down to kSortBucket members (or to the end, see kFewEntries), then the sorted
// kernel, the aligned walk and the register kernel as sort_from() and kSmallBucket say
template <class P, bool RG, bool ST, int NV>
int launch_doubles(sci_ctx *ctx, const Tabs &T, const typename P::TT *tab, const typename P::CI *C, int nvec, int v0,
                   typename P::TO *S, bool &chained)
{
    if (T.e2 == 0) return SCI_OK;
    const size_t per = NV * sizeof(typename P::SC) + row_extra<RG>();
    const sci::Split &sp = T.split(per);
    int rc = launch_tiled<P, RG, ST, NV>(ctx, T, sp, tab, C, nvec, v0, S, chained);
    // the entries from lo on of buckets of at most `maxb` members, up to hi
    auto aligned = [&](auto kern, int64_t lo, int64_t hi, int maxb, int rows) -> int {
        if (hi <= lo) return SCI_OK;
        size_t smem = 0;
        const int ch = choose_rows(maxb, per, smem, rows);
        if (ch < 0) return sci_fail(ctx, SCI_ERR_OVERFLOW, "bucket too large for shared memory");
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return sci_cuda_check(ctx, e, "cudaFuncSetAttribute");
        }
        cudaError_t e = launch_chained(chained, kern, dim3((unsigned)((hi - lo + ch - 1) / ch) + 1), smem, ctx->stream,
                                       T.e2_idx + lo, T.e2_code + lo, T.e2_pos + lo, hi - lo, ch, tab_rule(ctx), tab,
                                       C, nvec, v0, S, T.rr, ST ? ctx->det_inv2 + lo : nullptr);
        chained = true;
        return sci_cuda_check(ctx, e, "k_doubles_aligned launch");
    };
    constexpr int rows = f32_wide<P, NV>() ? SCI_F32_ROWS : kRowsPerCta;
    // the first entry of each part: the tiles end at b, the middle buckets at m, the sorted
    // ones at so, the aligned ones of five members and more at sm
    const int64_t *above = T.ts->above;
    const int64_t b = sp.big, large = std::max(b, above[kSortBucket]);
    const int64_t m = in_one_walk<P, RG>(T.e2, b, large) ? T.e2 : large;
    constexpr int lowest = sort_from<P, NV>(true);
    const int from = sort_from<P, NV>(ctx->tab_elems * (int64_t)sizeof(typename P::TT) <= kSmallTable);
    const int64_t sm = lowest <= kSmallBucket ? T.e2 : std::max(m, above[kSmallBucket]);
    const int64_t so = from > kSortBucket ? m : std::min(sm, std::max(m, above[from - 1]));
    if (rc == SCI_OK)
        rc = aligned(k_doubles_aligned<P, NV, RG, ST, wide_ctas<P, NV>()>, b, m, sp.maxb_small,
                     window_rows(m - b, rows));
    if (rc != SCI_OK) return rc;
    if constexpr (lowest <= kSortBucket) {
        if (so > m) {
            constexpr size_t smem = sort_smem<P, NV>();
            auto kern = k_doubles_sorted<P, NV, RG, ST>;
            if constexpr (smem > 47 * 1024) {   // static shared memory counts against the 48 KB too
                cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return sci_cuda_check(ctx, e, "cudaFuncSetAttribute");
            }
            cudaError_t e = launch_chained(chained, kern, dim3((unsigned)((so - m + kSortRows - 1) / kSortRows) + 1),
                                           smem, ctx->stream, T.e2_idx + m, T.e2_code + m, T.e2_pos + m, so - m,
                                           tab_rule(ctx), tab, C, nvec, v0, S, T.rr, ST ? ctx->det_inv2 + m : nullptr);
            chained = true;
            if ((rc = sci_cuda_check(ctx, e, "k_doubles_sorted launch")) != SCI_OK) return rc;
        }
    }
    if constexpr (lowest > kSmallBucket) {
        if constexpr (sort_from<P, NV>(false) > kSmallBucket + 1)
            rc = aligned(k_doubles_aligned<P, NV, RG, ST, min_ctas<P, NV>()>, so, sm, std::min(from - 1, sp.maxb_small),
                         rows);
        if (rc != SCI_OK) return rc;
        auto small = [&](auto kern, int size) -> int {   // the buckets of `size` members
            const int64_t lo = std::max(m, above[size]), hi = std::max(m, above[size - 1]);
            if (hi == lo) return SCI_OK;
            const int64_t nb = (hi - lo) / size;
            cudaError_t e = launch_chained(chained, kern, dim3((unsigned)((nb * NV + kThreads - 1) / kThreads) + 1), 0,
                                           ctx->stream, T.e2_idx + lo, T.e2_code + lo, nb, tab_rule(ctx), tab, C, nvec,
                                           v0, S, T.rr, ST ? ctx->det_inv2 + lo : nullptr);
            chained = true;
            return sci_cuda_check(ctx, e, "k_doubles_small launch");
        };
        rc = small(k_doubles_small<P, 4, NV, RG, ST>, 4);
        if (rc == SCI_OK) rc = small(k_doubles_small<P, 3, NV, RG, ST>, 3);
        if (rc == SCI_OK) rc = small(k_doubles_small<P, 2, NV, RG, ST>, 2);
    }
    return rc;
}

// paired-FP32 doubles: real (float2 table, float2 staged c) or complex (float4 / float4)
template <bool RG, bool ST, bool CPLX, int NV>
int launch_doubles_ds(sci_ctx *ctx, const Tabs &T, const void *C, void *S, int nvec, int v0)
{
    if (T.e2 == 0) return SCI_OK;
    // the vector group, split into paired floats in the context's c_ds buffer
    // (64 bytes per determinant: up to 8 real or 4 complex coefficients)
    if constexpr (CPLX)
        k_split_cz<<<grid_for(ctx->M * NV), kThreads, 0, ctx->stream>>>((const zdbl *)C, ctx->M, nvec, v0, NV,
                                                                        (float4 *)ctx->c_ds);
    else
        k_split_c<<<grid_for(ctx->M * NV), kThreads, 0, ctx->stream>>>((const double *)C, ctx->M, nvec, v0, NV,
                                                                       (float2 *)ctx->c_ds);
    SCI_CK(cudaGetLastError());
    bool chained = false;   // the first launch reads the split copy made just before
    if constexpr (CPLX)
        return launch_doubles<PolDSZ, RG, ST, NV>(ctx, T, (const float4 *)ctx->tab_ds, (const float4 *)ctx->c_ds, nvec, v0, (zdbl *)S, chained);
    else
        return launch_doubles<PolDS, RG, ST, NV>(ctx, T, (const float2 *)ctx->tab_ds, (const float2 *)ctx->c_ds, nvec, v0, (double *)S, chained);
}

template <bool RG, bool ST, bool CPLX>
int ds_groups(sci_ctx *ctx, const Tabs &T, const void *C, void *S, int nvec)
{
    int rc = SCI_OK;
    const size_t unit = CPLX ? sizeof(float4) : sizeof(float2);
    for (int v0 = 0; v0 < nvec && rc == SCI_OK;) {
        int left = nvec - v0;
        int g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        if (CPLX && g > 4) g = 4;
        size_t smem_probe = 0;
        while (g > 1 && choose_rows(T.maxb_small(), g * unit + row_extra<RG>(), smem_probe) < 0) g >>= 1;
        switch (g) {
        case 8:
            if constexpr (!CPLX) rc = launch_doubles_ds<RG, ST, CPLX, 8>(ctx, T, C, S, nvec, v0);
            break;
        case 4: rc = launch_doubles_ds<RG, ST, CPLX, 4>(ctx, T, C, S, nvec, v0); break;
        case 2: rc = launch_doubles_ds<RG, ST, CPLX, 2>(ctx, T, C, S, nvec, v0); break;
        default: rc = launch_doubles_ds<RG, ST, CPLX, 1>(ctx, T, C, S, nvec, v0); break;
        }
        v0 += g;
    }
    return rc;
}

// FP32-storage doubles (SCI_PREC_F32_STORE_F64_ACC)
template <bool RG, bool ST>
int f32_groups(sci_ctx *ctx, const Tabs &T, const float *C, double *S, int nvec)
{
    int rc = SCI_OK;
    bool chained = false;
    for (int v0 = 0; v0 < nvec && rc == SCI_OK;) {
        int left = nvec - v0;
        int g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        size_t smem_probe = 0;
        while (g > 1 && choose_rows(T.maxb_small(), g * sizeof(float) + row_extra<RG>(), smem_probe) < 0) g >>= 1;
        switch (g) {
        case 8: rc = launch_doubles<PolF32, RG, ST, 8>(ctx, T, ctx->tab32, C, nvec, v0, S, chained); break;
        case 4: rc = launch_doubles<PolF32, RG, ST, 4>(ctx, T, ctx->tab32, C, nvec, v0, S, chained); break;
        case 2: rc = launch_doubles<PolF32, RG, ST, 2>(ctx, T, ctx->tab32, C, nvec, v0, S, chained); break;
        default: rc = launch_doubles<PolF32, RG, ST, 1>(ctx, T, ctx->tab32, C, nvec, v0, S, chained); break;
        }
        v0 += g;
    }
    return rc;
}

// paired-FP32 singles; real coefficients may come in as double or float; keys of one to
// four words (KW)
template <bool RG, bool ST, bool CPLX, int NV, typename TC, int KW>
int launch_singles_ds_w(sci_ctx *ctx, const Tabs &T, const void *C, void *S, int nvec, int v0)
{
    const int g = grid_for(T.e1);
    if constexpr (CPLX) {
        k_split_cz<<<grid_for(ctx->M * NV), kThreads, 0, ctx->stream>>>((const zdbl *)C, ctx->M, nvec, v0, NV,
                                                                        (float4 *)ctx->c_ds);
        k_singles_dsz<NV, RG, ST, KW><<<g, kThreads, 0, ctx->stream>>>(
            T.e1_idx, T.e1_S, T.e1_meta, T.e1, ctx->norb, ref_words(ctx), (const float4 *)ctx->fref_ds,
            (const float4 *)ctx->g_ds, (const float4 *)ctx->c_ds, nvec, v0, (zdbl *)S, T.rr,
            ST ? ctx->det_inv1 : nullptr);
    } else {
        k_split_c<TC><<<grid_for(ctx->M * NV), kThreads, 0, ctx->stream>>>((const TC *)C, ctx->M, nvec, v0, NV,
                                                                           (float2 *)ctx->c_ds);
        k_singles_ds<NV, RG, ST, KW><<<g, kThreads, 0, ctx->stream>>>(
            T.e1_idx, T.e1_S, T.e1_meta, T.e1, ctx->norb, ref_words(ctx), (const float2 *)ctx->fref_ds,
            (const float2 *)ctx->g_ds, (const float2 *)ctx->c_ds, nvec, v0, (double *)S, T.rr,
            ST ? ctx->det_inv1 : nullptr);
    }
    return sci_cuda_check(ctx, cudaGetLastError(), "k_singles_ds launch");
}

template <bool RG, bool ST, bool CPLX, int NV, typename TC = double>
int launch_singles_ds(sci_ctx *ctx, const Tabs &T, const void *C, void *S, int nvec, int v0)
{
    if (T.e1 == 0) return SCI_OK;
    if (ctx->nwords == 4) return launch_singles_ds_w<RG, ST, CPLX, NV, TC, 4>(ctx, T, C, S, nvec, v0);
    if (ctx->nwords == 3) return launch_singles_ds_w<RG, ST, CPLX, NV, TC, 3>(ctx, T, C, S, nvec, v0);
    if (ctx->nwords == 2) return launch_singles_ds_w<RG, ST, CPLX, NV, TC, 2>(ctx, T, C, S, nvec, v0);
    return launch_singles_ds_w<RG, ST, CPLX, NV, TC, 1>(ctx, T, C, S, nvec, v0);
}

template <bool RG, bool ST, bool CPLX, typename TC = double>
int ds_singles_groups(sci_ctx *ctx, const Tabs &T, const void *C, void *S, int nvec)
{
    int rc = SCI_OK;
    for (int v0 = 0; v0 < nvec && rc == SCI_OK;) {
        int left = nvec - v0;
        int g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        if (CPLX && g > 4) g = 4;
        switch (g) {
        case 8:
            if constexpr (!CPLX) rc = launch_singles_ds<RG, ST, CPLX, 8, TC>(ctx, T, C, S, nvec, v0);
            break;
        case 4: rc = launch_singles_ds<RG, ST, CPLX, 4, TC>(ctx, T, C, S, nvec, v0); break;
        case 2: rc = launch_singles_ds<RG, ST, CPLX, 2, TC>(ctx, T, C, S, nvec, v0); break;
        default: rc = launch_singles_ds<RG, ST, CPLX, 1, TC>(ctx, T, C, S, nvec, v0); break;
        }
        v0 += g;
    }
    return rc;
}

template <bool RG, bool ST, typename TS, typename TC, int NV>
int launch_singles(sci_ctx *ctx, const Tabs &T, const TC *C, typename AccOf<TS>::type *S, int nvec, int v0, bool &chained)
{
    if (T.e1 == 0) return SCI_OK;
    auto kern = ctx->nwords == 4   ? k_singles<TS, TC, NV, RG, ST, 4>
                : ctx->nwords == 3 ? k_singles<TS, TC, NV, RG, ST, 3>
                : ctx->nwords == 2 ? k_singles<TS, TC, NV, RG, ST, 2>
                                   : k_singles<TS, TC, NV, RG, ST, 1>;
    cudaError_t e = launch_chained(chained, kern, dim3(grid_for(T.e1)), 0, ctx->stream, T.e1_idx, T.e1_S, T.e1_meta,
                                   T.e1, ctx->norb, ref_words(ctx), (const TS *)ctx->fref, (const TS *)ctx->g_so, C,
                                   nvec, v0, S, T.rr, ST ? ctx->det_inv1 : nullptr);
    chained = true;
    return sci_cuda_check(ctx, e, "k_singles launch");
}

template <bool RG, bool ST, typename TS, typename TC>
int sigma_groups(sci_ctx *ctx, const Tabs &T, const TS *tab, const TC *C, typename AccOf<TS>::type *S, int nvec,
                 bool &chained)
{
    int rc = SCI_OK;
    for (int v0 = 0; v0 < nvec && rc == SCI_OK;) {
        int left = nvec - v0;
        int g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        if (sizeof(TS) == 16 && g > 4) g = 4;
        size_t smem_probe = 0;  // shrink the vector group until its window fits
        while (g > 1 && choose_rows(T.maxb_small(), g * sizeof(TS) + row_extra<RG>(), smem_probe) < 0) g >>= 1;
        switch (g) {
        case 8:
            if constexpr (sizeof(TS) == sizeof(double))
                rc = launch_doubles<PolF64<TS, TC>, RG, ST, 8>(ctx, T, tab, C, nvec, v0, S, chained);
            break;
        case 4: rc = launch_doubles<PolF64<TS, TC>, RG, ST, 4>(ctx, T, tab, C, nvec, v0, S, chained); break;
        case 2: rc = launch_doubles<PolF64<TS, TC>, RG, ST, 2>(ctx, T, tab, C, nvec, v0, S, chained); break;
        default: rc = launch_doubles<PolF64<TS, TC>, RG, ST, 1>(ctx, T, tab, C, nvec, v0, S, chained); break;
        }
        v0 += g;
    }
    return rc;
}

template <bool RG, bool ST, typename TS, typename TC>
int singles_groups(sci_ctx *ctx, const Tabs &T, const TC *C, typename AccOf<TS>::type *S, int nvec, bool &chained)
{
    int rc = SCI_OK;
    for (int v0 = 0; v0 < nvec && rc == SCI_OK;) {
        int left = nvec - v0;
        int g = left >= 4 ? 4 : left >= 2 ? 2 : 1;
        switch (g) {
        case 4: rc = launch_singles<RG, ST, TS, TC, 4>(ctx, T, C, S, nvec, v0, chained); break;
        case 2: rc = launch_singles<RG, ST, TS, TC, 2>(ctx, T, C, S, nvec, v0, chained); break;
        default: rc = launch_singles<RG, ST, TS, TC, 1>(ctx, T, C, S, nvec, v0, chained); break;
        }
        v0 += g;
    }
    return rc;
}

// ------------------------------------------------------------------ pair counting
__global__ void k_count2(const uint32_t *__restrict__ e_code, const uint32_t *__restrict__ e_pos, int64_t E,
                         unsigned long long *out)
{
    unsigned long long cnt = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t pos = e_pos[p];
        const int64_t bs = p - sci::pos_off(pos), be = bs + sci::pos_size(pos);
        const uint32_t cp = e_code[p];
        for (int64_t q = bs; q < be; q++) cnt += !sci::codes_overlap(e_code[q], cp);
    }
    for (int o = 16; o; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(out, cnt);
}

__global__ void k_count1(const uint32_t *__restrict__ e_meta, int64_t E, unsigned long long *out)
{
    unsigned long long cnt = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x)
        cnt += sci::meta_size(e_meta[p]) - 1;
    for (int o = 16; o; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(out, cnt);
}

// ------------------------------------------------------------------ connection export
struct ConnOut {
    int64_t *row, *col;
    int8_t *deg, *ph;
    int64_t cap;
    unsigned long long *counter;
};

__device__ __forceinline__ void conn_put(ConnOut o, int64_t r, int64_t c, int d, int ph)
{
    unsigned long long s = atomicAdd(o.counter, 1ull);
    if ((int64_t)s < o.cap) {
        o.row[s] = r;
        o.col[s] = c;
        o.deg[s] = (int8_t)d;
        o.ph[s] = (int8_t)ph;
    }
}

__global__ void k_conn2(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code,
                        const uint32_t *__restrict__ e_pos, int64_t E, int64_t rb, int64_t re, ConnOut o)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t I = e_idx[p];
        if (I < rb || I >= re) continue;
        const uint32_t pos = e_pos[p], code = e_code[p];
        const int64_t bs = p - sci::pos_off(pos), be = bs + sci::pos_size(pos);
        const int par = sci::code_par(code);
        for (int64_t q = bs; q < be; q++) {
            const uint32_t cq = e_code[q];
            if (sci::codes_overlap(cq, code)) continue;
            conn_put(o, I, e_idx[q], 2, (par ^ (int)sci::code_par(cq)) ? -1 : 1);
        }
    }
}

__global__ void k_conn1(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_meta, int64_t E, int64_t rb,
                        int64_t re, ConnOut o)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x) {
        int64_t I = e_idx[p];
        if (I < rb || I >= re) continue;
        uint32_t meta = e_meta[p];
        int64_t bs = p - (int64_t)sci::meta_off(meta), be = bs + (int64_t)sci::meta_size(meta);
        int par = sci::meta_par(meta);
        for (int64_t q = bs; q < be; q++) {
            if (q == p) continue;
            int parq = sci::meta_par(e_meta[q]);
            conn_put(o, I, e_idx[q], 1, (par ^ parq) ? -1 : 1);
        }
    }
}

inline void mark(sci_ctx *ctx, int i)
{
    if (ctx->profile) cudaEventRecord(ctx->ev[i], ctx->stream);
}

}  // namespace

// whether the largest (N-2) bucket fits the staging window of a one-vector launch in the
// context's scalar mode, row-range launches included (wider vector groups shrink until
// they fit, down to one vector)
bool sci_sigma_window_fits(const sci_ctx *ctx)
{
    size_t smem = 0;
    const size_t per = (ctx->cplx ? sizeof(zdbl) : sizeof(double)) + row_extra<true>();
    return ctx->e2 == ctx->split2.base.big || choose_rows(ctx->split2.base.maxb_small, per, smem) >= 0;
}

namespace {

// Deterministic accumulation: S_I = H_II C_I + the row sums the double- and single-
// excitation kernels stored for row I's bucket entries.  They store them in row order (the
// slot of an entry is its position among the entries sorted by row), so row I's sums are
// the contiguous segment [ptr[I], ptr[I + 1]).  One warp per row: lane l adds the segment's
// elements l, l + 32, ..., then the lanes are combined by a fixed butterfly of shuffles,
// so the result does not depend on scheduling.
__device__ __forceinline__ void add_to(double &a, double b) { a += b; }
__device__ __forceinline__ void add_to(zdbl &a, zdbl b) { a.x += b.x, a.y += b.y; }
__device__ __forceinline__ double shfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ zdbl shfl_xor(zdbl a, int o)
{
    return zdbl{__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o)};
}
__device__ __forceinline__ double diag_times(double h, double c) { return h * c; }
__device__ __forceinline__ double diag_times(double h, float c) { return h * (double)c; }
__device__ __forceinline__ zdbl diag_times(double h, zdbl c) { return zdbl{h * c.x, h * c.y}; }

// Lanes per row of k_row_sums.  A row holds ~C(N,2)/2 + N slots on average (about 100 on
// the 20-electron spaces), so four lanes per row keep the lanes busy and the butterfly at
// two levels; a warp per row spent more FP64 adds on its butterfly and on padding than on
// the slots (2M-determinant space, one vector: 1.97 ms with a warp per row, FP64 pipe 83%
// busy in ncu; 0.80 ms with four lanes).
constexpr int kRowLanes = 4;

template <typename TC, typename TA, int NV>
__global__ void __launch_bounds__(kThreads)
k_row_sums(int64_t M, int nvec, int v0, const double *__restrict__ hdiag, const TC *__restrict__ C,
           const uint32_t *__restrict__ ptr2, const TA *__restrict__ part2, const uint32_t *__restrict__ ptr1,
           const TA *__restrict__ part1, TA *__restrict__ S)
{
    constexpr int G = kRowLanes, RPW = 32 / G;   // lanes per row, rows per warp
    const int lane = threadIdx.x & 31, gl = lane & (G - 1);
    const int64_t warps = (int64_t)gridDim.x * (kThreads / 32);
    // warp-uniform loop (the butterfly needs every lane); a lane past M adds nothing
    for (int64_t Ib = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / 32 * RPW; Ib < M; Ib += warps * RPW) {
        const int64_t I = Ib + lane / G;
        TA acc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) zero(acc[v]);
        if (I < M) {
            // the row's doubles slots, then its singles slots: lane gl adds slots gl, gl + G,
            // ... in order, four loads in flight per step, each add predicated on its slot
            for (int tab = 0; tab < 2; tab++) {
                const uint32_t *ptr = tab ? ptr1 : ptr2;
                const TA *part = tab ? part1 : part2;
                const uint32_t end = ptr[I + 1];
                for (uint32_t t0 = ptr[I] + gl; t0 < end; t0 += 4 * G) {
                    TA x[4][NV];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const uint32_t t = t0 + G * u;
                        const TA *src = part + (int64_t)t * nvec + v0;
#pragma unroll
                        for (int v = 0; v < NV; v++) {
                            zero(x[u][v]);
                            if (t < end) x[u][v] = src[v];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (t0 + G * u < end)
#pragma unroll
                            for (int v = 0; v < NV; v++) add_to(acc[v], x[u][v]);
                }
            }
        }
#pragma unroll
        for (int v = 0; v < NV; v++)
#pragma unroll
            for (int o = G / 2; o; o >>= 1) add_to(acc[v], shfl_xor(acc[v], o));
        if (I < M) {
            // lane gl writes vectors gl, gl + G, ...: H_II c_I plus the row sum
#pragma unroll
            for (int v = 0; v < NV; v++)
                if (v % G == gl) {
                    TA out = diag_times(hdiag[I], C[I * nvec + v0 + v]);
                    add_to(out, acc[v]);
                    S[I * nvec + v0 + v] = out;
                }
        }
    }
}

template <typename TC, typename TA>
int row_sums(sci_ctx *ctx, const TC *C, TA *S, int nvec)
{
    const int64_t M = ctx->M;
    const int grid = grid_for(M * kRowLanes);
    auto go = [&](auto kern, int v0) {
        kern<<<grid, kThreads, 0, ctx->stream>>>(M, nvec, v0, ctx->hdiag, C, ctx->det_ptr2, (const TA *)ctx->det_part2,
                                                 ctx->det_ptr1, (const TA *)ctx->det_part1, S);
    };
    for (int v0 = 0; v0 < nvec;) {
        const int left = nvec - v0;
        const int g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        switch (g) {
        case 8: go(k_row_sums<TC, TA, 8>, v0); break;
        case 4: go(k_row_sums<TC, TA, 4>, v0); break;
        case 2: go(k_row_sums<TC, TA, 2>, v0); break;
        default: go(k_row_sums<TC, TA, 1>, v0); break;
        }
        v0 += g;
    }
    return sci_cuda_check(ctx, cudaGetLastError(), "k_row_sums launch");
}

// one sigma launch sequence over the tables T (RG: the rows of a row range only; ST: the
// deterministic accumulation, row sums stored in the entries' slots, then per-row sums)
template <bool RG, bool ST>
int launch_sigma(sci_ctx *ctx, const Tabs &T, const void *C, void *S_out, int nvec, int prec)
{
    // with ST the double- and single-excitation kernels write the slots, not S
    void *S = ST ? ctx->det_part2 : S_out;
    void *S1 = ST ? ctx->det_part1 : S_out;
    cudaStream_t st = ctx->stream;
    const int64_t row0 = T.rr.rb, nrows = T.rr.re - T.rr.rb;
    int rc;
    bool chained = false;   // whether a launch of the FP64 chain precedes
    mark(ctx, 0);
    if (ctx->cplx) {
        const zdbl *Cz = (const zdbl *)C;
        zdbl *Sz = (zdbl *)S;
        if (!ST && nrows > 0)
            k_sigma_init<zdbl, zdbl><<<grid_for(nrows * nvec), kThreads, 0, st>>>(ctx->hdiag, Cz, Sz, row0, nrows, nvec);
        SCI_CK(cudaGetLastError());
        mark(ctx, 1);
        rc = prec == SCI_PREC_F64_DS ? ds_groups<RG, ST, true>(ctx, T, C, S, nvec)
                                     : sigma_groups<RG, ST, zdbl, zdbl>(ctx, T, (const zdbl *)ctx->tab, Cz, Sz, nvec, chained);
        mark(ctx, 2);
        if (rc == SCI_OK)
            rc = prec == SCI_PREC_F64_DS ? ds_singles_groups<RG, ST, true>(ctx, T, C, S1, nvec)
                                         : singles_groups<RG, ST, zdbl, zdbl>(ctx, T, Cz, (zdbl *)S1, nvec, chained);
        mark(ctx, 3);
        if (ST && rc == SCI_OK) rc = row_sums<zdbl, zdbl>(ctx, Cz, (zdbl *)S_out, nvec);
        mark(ctx, 4);
        return rc;
    }
    double *Sd = (double *)S;
    if (prec == SCI_PREC_F64 || prec == SCI_PREC_F64_DS) {
        const double *Cd = (const double *)C;
        if (!ST && nrows > 0)
            k_sigma_init<double, double><<<grid_for(nrows * nvec), kThreads, 0, st>>>(ctx->hdiag, Cd, Sd, row0, nrows,
                                                                                       nvec);
        SCI_CK(cudaGetLastError());
        mark(ctx, 1);
        rc = prec == SCI_PREC_F64_DS ? ds_groups<RG, ST, false>(ctx, T, C, S, nvec)
                                     : sigma_groups<RG, ST, double, double>(ctx, T, (const double *)ctx->tab, Cd, Sd, nvec, chained);
        mark(ctx, 2);
        if (rc == SCI_OK)
            rc = prec == SCI_PREC_F64_DS ? ds_singles_groups<RG, ST, false>(ctx, T, C, S1, nvec)
                                         : singles_groups<RG, ST, double, double>(ctx, T, Cd, (double *)S1, nvec, chained);
        mark(ctx, 3);
        if (ST && rc == SCI_OK) rc = row_sums<double, double>(ctx, Cd, (double *)S_out, nvec);
        mark(ctx, 4);
        return rc;
    }
    const float *Cf = (const float *)C;
    if (!ST && nrows > 0)
        k_sigma_init<float, double><<<grid_for(nrows * nvec), kThreads, 0, st>>>(ctx->hdiag, Cf, Sd, row0, nrows, nvec);
    SCI_CK(cudaGetLastError());
    mark(ctx, 1);
    rc = f32_groups<RG, ST>(ctx, T, Cf, Sd, nvec);
    mark(ctx, 2);
    if (rc == SCI_OK) rc = ds_singles_groups<RG, ST, false, float>(ctx, T, C, S1, nvec);
    mark(ctx, 3);
    if (ST && rc == SCI_OK) rc = row_sums<float, double>(ctx, Cf, (double *)S_out, nvec);
    mark(ctx, 4);
    return rc;
}

}  // namespace

int sci_launch_sigma(sci_ctx *ctx, const void *C, void *S, int nvec, int prec, bool whole_list)
{
    if (whole_list || !ctx->ranged) {
        const bool ranged = ctx->ranged;
        ctx->ranged = 0;   // tabs_of: the full tables
        const Tabs T = tabs_of(ctx);
        ctx->ranged = ranged;
        if (ctx->det_nvec > 0 && nvec <= ctx->det_nvec) return launch_sigma<false, true>(ctx, T, C, S, nvec, prec);
        return launch_sigma<false, false>(ctx, T, C, S, nvec, prec);
    }
    return launch_sigma<true, false>(ctx, tabs_of(ctx), C, S, nvec, prec);
}

int sci_count_pairs_device(sci_ctx *ctx, int64_t *pairs2, int64_t *pairs1)
{
    cudaStream_t st = ctx->stream;
    unsigned long long *d = nullptr;
    SCI_CK(cudaMalloc(&d, 16));
    cudaMemsetAsync(d, 0, 16, st);
    if (ctx->e2 > 0) k_count2<<<grid_for(ctx->e2), kThreads, 0, st>>>(ctx->e2_code, ctx->e2_pos, ctx->e2, d);
    if (ctx->e1 > 0) k_count1<<<grid_for(ctx->e1), kThreads, 0, st>>>(ctx->e1_meta, ctx->e1, d + 1);
    unsigned long long h[2] = {0, 0};
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, 16, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    SCI_CK(e);
    *pairs2 = (int64_t)h[0];
    *pairs1 = (int64_t)h[1];
    return SCI_OK;
}

int sci_connections_device(sci_ctx *ctx, int64_t row_begin, int64_t row_end, int64_t *count, int64_t *rows,
                           int64_t *J, int8_t *degree, int8_t *phase, int64_t cap)
{
    cudaStream_t st = ctx->stream;
    unsigned long long *counter = nullptr;
    SCI_CK(cudaMalloc(&counter, 8));
    // pass 1: count
    ConnOut o{nullptr, nullptr, nullptr, nullptr, 0, counter};
    cudaMemsetAsync(counter, 0, 8, st);
    if (ctx->e2 > 0)
        k_conn2<<<grid_for(ctx->e2), kThreads, 0, st>>>(ctx->e2_idx, ctx->e2_code, ctx->e2_pos, ctx->e2, row_begin,
                                                         row_end, o);
    if (ctx->e1 > 0)
        k_conn1<<<grid_for(ctx->e1), kThreads, 0, st>>>(ctx->e1_idx, ctx->e1_meta, ctx->e1, row_begin, row_end, o);
    unsigned long long n = 0;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&n, counter, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { cudaFree(counter); return sci_cuda_check(ctx, e, "connection count"); }
    *count = (int64_t)n;
    if ((int64_t)n > cap) { cudaFree(counter); return sci_fail(ctx, SCI_ERR_OVERFLOW, "connection list exceeds cap"); }
    if (n == 0) { cudaFree(counter); return SCI_OK; }
    // pass 2: fill
    void *buf = nullptr;
    e = cudaMalloc(&buf, n * 18);
    if (e != cudaSuccess) { cudaFree(counter); return sci_cuda_check(ctx, e, "connection buffer"); }
    o.row = (int64_t *)buf;
    o.col = o.row + n;
    o.deg = (int8_t *)(o.col + n);
    o.ph = o.deg + n;
    o.cap = (int64_t)n;
    cudaMemsetAsync(counter, 0, 8, st);
    if (ctx->e2 > 0)
        k_conn2<<<grid_for(ctx->e2), kThreads, 0, st>>>(ctx->e2_idx, ctx->e2_code, ctx->e2_pos, ctx->e2, row_begin,
                                                         row_end, o);
    if (ctx->e1 > 0)
        k_conn1<<<grid_for(ctx->e1), kThreads, 0, st>>>(ctx->e1_idx, ctx->e1_meta, ctx->e1, row_begin, row_end, o);
    std::vector<int64_t> hr(n), hc(n);
    std::vector<int8_t> hd(n), hp(n);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(hr.data(), o.row, n * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hc.data(), o.col, n * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hd.data(), o.deg, n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hp.data(), o.ph, n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(buf);
    cudaFree(counter);
    SCI_CK(e);
    std::vector<int64_t> perm(n);
    for (size_t t = 0; t < n; t++) perm[t] = (int64_t)t;
    std::sort(perm.begin(), perm.end(), [&](int64_t a, int64_t b) {
        return hr[a] != hr[b] ? hr[a] < hr[b] : hc[a] < hc[b];
    });
    for (size_t t = 0; t < n; t++) {
        int64_t s = perm[t];
        if (rows) rows[t] = hr[s];
        if (J) J[t] = hc[s];
        if (degree) degree[t] = hd[s];
        if (phase) phase[t] = hp[s];
    }
    return SCI_OK;
}
