// Reduced density matrices (Sec. 3.4) by the same bucket walks as sigma.
//
//   g1[p][q]       = sum_k w_k <c_k| a+_p a_q |c_k>
//   g2[p][q][r][s] = sum_k w_k <c_k| a+_p a+_r a_s a_q |c_k>
// over spin-orbitals (bit order of the keys) or spinors, unnormalised, so that for a
// normalised c the energy of Eq. Hamiltonian is sum h g1 + 1/2 sum (pq|rs) g2.
//
// The connections are recomputed from the setup tables, never stored.  The pairs of the
// three Slater-Condon classes (Sec. 2.3: zero, one and two differences) touch disjoint
// sets of g2 elements, so each class is accumulated into its own compact table and
// expanded once at the end:
//   diagonal (I = J): g1[p][p] and g2[p][p][r][r] = -g2[p][r][r][p] = sum_I w_I n_p n_r.
//     With n(I) = n(ref) + Delta(I) (Delta nonzero on the <= 2 x level orbitals where I
//     and the reference differ) the pair occupation is
//       O[p][r] = Wt n_p n_r + n_p D_r + D_p n_r + DD[p][r],
//     Wt = sum w_I, D = sum w_I Delta(I), DD = sum w_I Delta Delta^T,
//     accumulated per CTA in shared memory.
//   singles (members X = S + x, Y = S + y of one (N-1) bucket): w = conj(c_X) c_Y ph,
//     g1[x][y] += w, and for every spectator k in S (A and Bc below take every unordered
//     pair in one orientation, and the expansion adds the conjugate)
//       g2[x][y][k][k] = g2[k][k][x][y] = -g2[x][k][k][y] = -g2[k][y][x][k] += w.
//     The spectator sum b[x][y][k] = sum w n_k(S) is kept as A[x][y] n_k(ref) + Bc[x][y][k]
//     with Bc taking only the orbitals of S that differ from the reference (the same
//     reference decomposition as the sigma singles).
//   doubles (members I = K + {a,b}, J = K + {i,j} of one (N-2) bucket, disjoint): one
//     atomic add of w = conj(c_I) c_J ph into a table laid out like the pair-integral
//     table (with separate alpha-alpha and beta-beta regions), every unordered pair in one
//     of its two orientations; the other is its conjugate.  Then
//       g2[a][i][b][j] = g2[b][j][a][i] = -g2[a][j][b][i] = -g2[b][i][a][j]
//         = dT[bra, ket] + conj(dT[ket, bra]).
// Signs: <I| a+_a a+_b a_j a_i |J> is the phase (-1)^(pi_I + pi_J) of the sigma kernels.
#include <algorithm>
#include <vector>

#include "sci_bits.cuh"
#include "sci_bucket.cuh"
#include "sci_internal.cuh"

using sci::zdbl;

namespace {

constexpr int kThreads = 256;
constexpr int kMaxVec = 8;  // vectors per walk; wider blocks take several walks

using sci::sflip;
__device__ __forceinline__ double conjv(double a) { return a; }
__device__ __forceinline__ zdbl conjv(zdbl a) { return zdbl{a.x, -a.y}; }
__device__ __forceinline__ double sqnorm(double a) { return a * a; }
__device__ __forceinline__ double sqnorm(zdbl a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ double scale(double a, double s) { return a * s; }
__device__ __forceinline__ zdbl scale(zdbl a, double s) { return zdbl{a.x * s, a.y * s}; }
__device__ __forceinline__ void zero(double &a) { a = 0.0; }
__device__ __forceinline__ void zero(zdbl &a) { a = zdbl{0.0, 0.0}; }
// a += x * y
__device__ __forceinline__ void mac(double &a, double x, double y) { a = fma(x, y, a); }
__device__ __forceinline__ void mac(zdbl &a, zdbl x, zdbl y)
{
    a.x = fma(x.x, y.x, fma(-x.y, y.y, a.x));
    a.y = fma(x.x, y.y, fma(x.y, y.x, a.y));
}
__device__ __forceinline__ double mul(double x, double y) { return x * y; }
__device__ __forceinline__ zdbl mul(zdbl x, zdbl y)
{
    return zdbl{fma(x.x, y.x, -x.y * y.y), fma(x.x, y.y, x.y * y.x)};
}
__device__ __forceinline__ void red(double *p, double v) { atomicAdd(p, v); }
__device__ __forceinline__ void red(zdbl *p, zdbl v)
{
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ zdbl neg(zdbl a) { return zdbl{-a.x, -a.y}; }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
template <typename TC> __device__ __forceinline__ TC from_real(double v);
template <> __device__ __forceinline__ double from_real<double>(double v) { return v; }
template <> __device__ __forceinline__ zdbl from_real<zdbl>(double v) { return zdbl{v, 0.0}; }
__device__ __forceinline__ zdbl add(zdbl a, zdbl b) { return zdbl{a.x + b.x, a.y + b.y}; }

// gradient-table offsets: the pair-table offsets, with beta-beta pairs moved to a region
// of their own after the alpha-alpha one (real spin-orbital mode)
__device__ __forceinline__ void grad_offsets(sci::TabRule tr, int x, int y, uint32_t bb_off, uint32_t &rowoff,
                                             uint32_t &colbase)
{
    sci::pair_offsets(tr, x, y, rowoff, colbase);
    if (!tr.spinors && x >= tr.n) colbase += bb_off;
}

// ------------------------------------------------------------------ diagonal
// occupation strings of KW 64-bit words: word w holds orbitals 64 w .. 64 w + 63
template <int KW> struct Str {
    uint64_t w[KW];
};
template <int KW> __device__ __forceinline__ Str<KW> load_str(const uint64_t *keys, int64_t I)
{
    Str<KW> s;
#pragma unroll
    for (int k = 0; k < KW; k++) s.w[k] = keys[I * KW + k];
    return s;
}
template <int KW> __device__ __forceinline__ bool occ(const Str<KW> &s, int p)
{
    return (s.w[p >> 6] >> (p & 63)) & 1;
}
using sci::RefW;   // the reference string over all words

// Diagonal class: O[p][r] = sum_I w_I n_p n_r in the reference decomposition n = n_ref + d
// (d = key ^ ref has a few bits, +1 on particles and -1 on holes), accumulated per CTA in
// shared memory ([norb]^2 doubles, dynamic: up to 226 KB, 168 spin-orbitals) when SM, else
// straight into DD and D in global memory (more orbitals).  Only DD[p][r] with p < r is kept;
// DD[p][p] = sum w d_p^2 is D[p] up to the sign of d_p.
//
// An FP64 add to shared memory is a compare-and-swap loop, and neighbouring determinants
// differ from the reference on the same orbitals.  So a warp takes its 32 determinants one
// after another, its lanes on the (p, r) pairs of one of them, all different addresses.
// 30 orbitals, M = 250k: a determinant per thread 399 us, a determinant per warp 149 us.
template <typename TC, int KW, bool SM = true>
__global__ void __launch_bounds__(kThreads)
k_rdm_diag(const uint64_t *__restrict__ keys, int64_t M, int norb, RefW ref,
           const TC *__restrict__ C, int nvec, int v0, int nv, const double *__restrict__ wk, double *__restrict__ Wt,
           double *__restrict__ D, double *__restrict__ DD)
{
    extern __shared__ double s_dyn[];
    __shared__ double s_wsum[kThreads / 32];
    __shared__ uint8_t s_orb[kThreads / 32][64 * KW];   // orbitals of a determinant outside the reference or missing
    double *sDD = SM ? s_dyn : DD, *sD = SM ? s_dyn + norb * norb : D;
    if constexpr (SM) {
        for (int i = threadIdx.x; i < norb * norb; i += blockDim.x) sDD[i] = 0.0;
        for (int i = threadIdx.x; i < norb; i += blockDim.x) sD[i] = 0.0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint8_t *orb = s_orb[wid];
    double wsum = 0.0;
    for (int64_t I0 = blockIdx.x * (int64_t)blockDim.x + 32 * wid; I0 < M; I0 += (int64_t)gridDim.x * blockDim.x) {
        const int cnt = (int)min((int64_t)32, M - I0);
        double wl = 0.0;
        Str<KW> mine{};
        if (lane < cnt) {
            const int64_t I = I0 + lane;
            for (int v = 0; v < nv; v++) wl = fma(wk[v0 + v], sqnorm(C[I * nvec + v0 + v]), wl);
            mine = load_str<KW>(keys, I);
        }
        wsum += wl;
        for (int u = 0; u < cnt; u++) {
            const double w = __shfl_sync(0xffffffffu, wl, u);
            int nd = 0;
#pragma unroll
            for (int k = 0; k < KW; k++) {
                const uint64_t m = __shfl_sync(0xffffffffu, (unsigned long long)mine.w[k], u) ^ ref.w[k];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const uint32_t mh = (uint32_t)(m >> (32 * h));
                    if ((mh >> lane) & 1u) orb[nd + __popc(mh & ((1u << lane) - 1u))] = (uint8_t)(64 * k + 32 * h + lane);
                    nd += __popc(mh);
                }
            }
            __syncwarp();
            for (int t = lane; t < nd * (nd + 1) / 2; t += 32) {   // t = b(b+1)/2 + a, a <= b
                int b = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
                while (b * (b + 1) / 2 > t) b--;
                while ((b + 1) * (b + 2) / 2 <= t) b++;
                const int p = orb[t - b * (b + 1) / 2], r = orb[b];
                const bool hp = (ref.w[p >> 6] >> (p & 63)) & 1, hr = (ref.w[r >> 6] >> (r & 63)) & 1;
                if (p == r) atomicAdd(&sD[p], sflip(hp, w));
                else atomicAdd(&sDD[p * norb + r], sflip(hp != hr, w));
            }
            __syncwarp();
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, off);
    if (lane == 0) s_wsum[wid] = wsum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < kThreads / 32; i++) t += s_wsum[i];
        atomicAdd(Wt, t);
    }
    if constexpr (SM) {
        for (int i = threadIdx.x; i < norb * norb; i += blockDim.x)
            if (sDD[i] != 0.0) atomicAdd(DD + i, sDD[i]);
        for (int i = threadIdx.x; i < norb; i += blockDim.x)
            if (sD[i] != 0.0) atomicAdd(D + i, sD[i]);
    }
}

// ------------------------------------------------------------------ pairs of a bucket
// Each unordered pair of a bucket of size s is walked once, with balanced work per row: the
// member at position q takes the members at q + d (mod s) for d = 1 .. ahead(q, s), which is
// (s-1)/2, and for even s one more in the first half of the bucket.  The orientation of a
// pair does not matter: the expansion adds both orientations.
__device__ __forceinline__ int ahead(int q, int s) { return (s - 1) / 2 + ((s & 1) == 0 && q < s / 2 ? 1 : 0); }

// ------------------------------------------------------------------ singles
// Bound by the FP64 atomic adds, 2 x level + 2 a pair, so a pair is walked once and not in both
// orders (30 orbitals, M = 250k, four vectors: 281 -> 148 us).
template <typename TC, int NV, int KW>
__global__ void __launch_bounds__(kThreads)
k_rdm_singles(const uint32_t *__restrict__ e_idx, const uint64_t *__restrict__ e_S, const uint32_t *__restrict__ e_meta,
              int64_t E, int norb, RefW ref, const TC *__restrict__ C, int nvec, int v0,
              const double *__restrict__ wk, TC *__restrict__ A, TC *__restrict__ Bc)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < E; p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t meta = e_meta[p];
        const int x = sci::meta_x(meta);
        const bool par = sci::meta_par(meta);
        const int off = sci::meta_off(meta), size = sci::meta_size(meta), na = ahead(off, size);
        if (na == 0) continue;
        // the spectator string's orbitals outside (part) and missing from (holes) the
        // reference, per word
        uint64_t part[KW], holes[KW];
#pragma unroll
        for (int k = 0; k < KW; k++) {
            const uint64_t Sk = e_S[p * KW + k], rk = ref.w[k];
            part[k] = Sk & ~rk, holes[k] = rk & ~Sk;
        }
        const int64_t idx = e_idx[p];
        TC rowc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) rowc[v] = scale(conjv(sflip(par, C[idx * nvec + v0 + v])), wk[v0 + v]);
        for (int d = 1; d <= na; d++) {
            const int64_t q = p + d - (off + d >= size ? size : 0);
            const uint32_t mq = e_meta[q];
            const int y = sci::meta_x(mq);
            const bool parq = sci::meta_par(mq);
            const int64_t idxq = e_idx[q];
            TC w;
            zero(w);
#pragma unroll
            for (int v = 0; v < NV; v++) mac(w, rowc[v], sflip(parq, C[idxq * nvec + v0 + v]));
            const int64_t xy = (int64_t)x * norb + y;
            red(A + xy, w);
            const TC nw = neg(w);
#pragma unroll
            for (int k = 0; k < KW; k++) {
                for (uint64_t m = part[k]; m; m &= m - 1) red(Bc + xy * norb + 64 * k + (__ffsll((long long)m) - 1), w);
                for (uint64_t m = holes[k]; m; m &= m - 1) red(Bc + xy * norb + 64 * k + (__ffsll((long long)m) - 1), nw);
            }
        }
    }
}

// ------------------------------------------------------------------ doubles
// A pair costs NV FP64 FMAs and one FP64 atomic add to the L2, and the FP64 pipe binds (a warp
// instruction holds it 16 cycles whatever its active lanes).  So the rows find their doubles
// first, as bit masks, and issue FP64 work for doubles only; by bucket size (entries are
// ordered by it, as in sigma): above kSortBucket members k_rdm_doubles, whose rows walk whole
// buckets and have similar counts; 5 to 64 k_rdm_doubles_sorted, rows sorted by their count;
// up to 4 k_rdm_doubles_small, in registers.
// 30 orbitals, M = 250k, four vectors: all sizes in one walk member by member 1.11 ms; 0.93 by
// size (above 64 members 0.49 ms, 5 to 64 0.35, up to 4 0.09).
constexpr int kMaskWords = 4;   // members per pass of a row over its bucket: 128

template <typename TC, int NV>
__global__ void __launch_bounds__(kThreads)
k_rdm_doubles(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code, const uint32_t *__restrict__ e_pos,
              int64_t E, int CH, sci::TabRule tr, uint32_t bb_off, const TC *__restrict__ C, int nvec, int v0,
              const double *__restrict__ wk, TC *__restrict__ dT)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_mask[kMaskWords][kThreads];   // a column per thread, no barrier needed
    int64_t r0, r1;
    sci::window(e_pos, E, CH, r0, r1);
    if (r0 >= r1) return;
    const int W = (int)(r1 - r0);
    TC *s_c = reinterpret_cast<TC *>(smem);  // [W][NV]: c of each member times (-1)^pi
    uint32_t *s_code = reinterpret_cast<uint32_t *>(s_c + (size_t)W * NV), *s_col = s_code + W;
    for (int q = threadIdx.x; q < W; q += blockDim.x) {
        const int64_t g = r0 + q;
        const uint32_t code = e_code[g];
        const int64_t idx = e_idx[g];
        uint32_t rowoff, colbase;
        grad_offsets(tr, sci::code_x(code), sci::code_y(code), bb_off, rowoff, colbase);
        s_code[q] = sci::col_code(code);
        s_col[q] = colbase;
        const bool par = sci::code_par(code);
        for (int v = 0; v < NV; v++) s_c[q * NV + v] = sflip(par, C[idx * nvec + v0 + v]);
    }
    __syncthreads();
    for (int q0 = threadIdx.x; q0 < W; q0 += blockDim.x) {
        const uint32_t code = e_code[r0 + q0], pos = e_pos[r0 + q0];
        uint32_t rowoff, colbase;
        grad_offsets(tr, sci::code_x(code), sci::code_y(code), bb_off, rowoff, colbase);
        const int qp = sci::pos_off(pos), sz = sci::pos_size(pos), bs = q0 - qp, be = bs + sz;
        const uint32_t rc = sci::row_code(code);
        TC rowc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) rowc[v] = scale(conjv(s_c[q0 * NV + v]), wk[v0 + v]);
        TC *trow = dT + rowoff;
        int at = q0 + 1, left = ahead(qp, sz);   // at: window row of the next member, before wrapping
        for (; left > 0; at += 32 * kMaskWords, left -= 32 * kMaskWords) {
            int n = 0;
            for (int w = 0; w < kMaskWords && 32 * w < left; w++) {
                const int j0 = at + 32 * w, len = min(32, left - 32 * w);
                // the members before and after the wrap to the start of the bucket
                const int first = min(max(be - j0, 0), len);
                uint32_t m = sci::doubles_mask(rc, s_code + j0, first);
                if (first < len) m |= sci::doubles_mask(rc, s_code + (j0 + first - sz), len - first) << first;
                s_mask[w][threadIdx.x] = m;
                n += __popc(m);
            }
            int w = -1;
            uint32_t m = 0;
            for (; n > 0; n--) {
                while (m == 0) m = s_mask[++w][threadIdx.x];
                int j = at + 32 * w + __ffs((int)m) - 1;
                m &= m - 1;
                j = j >= be ? j - sz : j;
                TC sum = mul(rowc[0], s_c[j * NV]);
#pragma unroll
                for (int v = 1; v < NV; v++) mac(sum, rowc[v], s_c[j * NV + v]);
                red(trow + s_col[j], sum);
            }
        }
    }
}

// Buckets of at most kSortBucket members.  A CTA owns the whole buckets that start in its
// kSortRows table rows; the doubles ahead of a row are a 64-bit mask, and the rows are sorted
// by their count, so that the lanes of a warp stay on useful products.  Members without any
// double read no coefficients.
constexpr int kSortRows = 448;
constexpr int kSortCap = kSortRows + sci::kSortBucket;   // rows of a window, at most
constexpr int kSortRounds = kSortCap / kThreads;
static_assert(kSortCap % kThreads == 0, "every thread holds the same number of rows");

template <typename TC, int NV> constexpr size_t sort_smem()
{
    return (size_t)kSortCap * (NV * sizeof(TC) + sizeof(uint64_t) + 3 * sizeof(uint32_t));
}

template <typename TC, int NV>
__global__ void __launch_bounds__(kThreads)
k_rdm_doubles_sorted(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code,
                     const uint32_t *__restrict__ e_pos, int64_t E, sci::TabRule tr, uint32_t bb_off,
                     const TC *__restrict__ C, int nvec, int v0, const double *__restrict__ wk, TC *__restrict__ dT)
{
    constexpr int kWarps = kThreads / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint16_t s_hist[kWarps][64];
    __shared__ int s_base[64], s_total;
    int64_t r0, r1;
    sci::window(e_pos, E, kSortRows, r0, r1);
    if (r0 >= r1) return;
    const int W = (int)(r1 - r0);
    TC *s_c = reinterpret_cast<TC *>(smem);
    uint64_t *s_mask = reinterpret_cast<uint64_t *>(s_c + kSortCap * NV);
    uint32_t *s_code = reinterpret_cast<uint32_t *>(s_mask + kSortCap);
    uint32_t *s_col = s_code + kSortCap;
    uint32_t *s_row = s_col + kSortCap;    // sorted rows: window row | bucket position << 16
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // warp w holds the rows [w * per, (w + 1) * per), 32 at a time
    const int per = ((W + kWarps - 1) / kWarps + 31) & ~31;

    uint32_t pos[kSortRounds];
    bool par[kSortRounds];
#pragma unroll
    for (int k = 0; k < kSortRounds; k++) {
        const int q = wid * per + 32 * k + lane;
        pos[k] = 0;
        par[k] = false;
        if (32 * k < per && q < W) {
            const uint32_t code = e_code[r0 + q];
            pos[k] = e_pos[r0 + q];
            par[k] = sci::code_par(code);
            uint32_t rowoff, colbase;
            grad_offsets(tr, sci::code_x(code), sci::code_y(code), bb_off, rowoff, colbase);
            s_code[q] = sci::col_code(code);
            s_col[q] = colbase;
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
            const int size = sci::pos_size(pos[k]), qp = sci::pos_off(pos[k]), bs = q - qp;
            const uint32_t rc = __byte_perm(s_code[q], 0, 0x1010);   // (x, y, x, y) of the row
            uint64_t m = sci::doubles_mask(rc, s_code + bs, min(size, 32));
            if (size > 32) m |= (uint64_t)sci::doubles_mask(rc, s_code + bs + 32, size - 32) << 32;
            if (m) {
                const int64_t I = e_idx[r0 + q];
#pragma unroll
                for (int v = 0; v < NV; v++) s_c[q * NV + v] = sflip(par[k], C[I * nvec + v0 + v]);
            }
            // the members ahead of the row, cyclically: bits qp + 1 .. qp + ahead (mod size)
            const uint64_t a = (1ull << ahead(qp, size)) - 1;
            const uint64_t window = (qp < 63 ? a << (qp + 1) : 0ull) | a >> (size - qp - 1);
            m &= window;   // bits from `size` on are no members and not set in m
            s_mask[q] = m;
            if (m) key[k] = 32 - __popcll(m);
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
            s_row[s_base[key[k]] + s_hist[wid][key[k]] + rank[k]] = (uint32_t)q | (uint32_t)sci::pos_off(pos[k]) << 16;
        }
    __syncthreads();

    const int nrows = s_total;
    for (int t = threadIdx.x; t < nrows; t += kThreads) {
        const uint32_t row = s_row[t];
        const int q = (int)(row & 0xFFFFu), bs = q - (int)(row >> 16);
        const uint32_t cc = s_code[q];
        uint32_t rowoff, colbase;
        grad_offsets(tr, (int)(cc & 0xFFu), (int)((cc >> 8) & 0xFFu), bb_off, rowoff, colbase);
        TC rowc[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) rowc[v] = scale(conjv(s_c[q * NV + v]), wk[v0 + v]);
        TC *trow = dT + rowoff;
        for (uint64_t m = s_mask[q]; m; m &= m - 1) {
            const int j = bs + __ffsll((long long)m) - 1;
            TC sum = mul(rowc[0], s_c[j * NV]);
#pragma unroll
            for (int v = 1; v < NV; v++) mac(sum, rowc[v], s_c[j * NV + v]);
            red(trow + s_col[j], sum);
        }
    }
}

// Buckets of S <= kSmallBucket members: most entries of a selected space, few of its pairs.  A
// thread takes a bucket, its members in registers; members without a double read nothing.
template <typename TC, int S, int NV>
__global__ void __launch_bounds__(kThreads)
k_rdm_doubles_small(const uint32_t *__restrict__ e_idx, const uint32_t *__restrict__ e_code, int64_t nbuckets,
                    sci::TabRule tr, uint32_t bb_off, const TC *__restrict__ C, int nvec, int v0,
                    const double *__restrict__ wk, TC *__restrict__ dT)
{
    const int64_t b = blockIdx.x * (int64_t)kThreads + threadIdx.x;
    if (b >= nbuckets) return;
    const int64_t g = b * S;
    uint32_t code[S], col[S];
    int64_t idx[S];
#pragma unroll
    for (int i = 0; i < S; i++) code[i] = e_code[g + i];
    bool any = false, dbl[S][S];
#pragma unroll
    for (int i = 0; i < S; i++)
#pragma unroll
        for (int j = 0; j < i; j++) {
            dbl[i][j] = sci::disjoint(sci::row_code(code[i]), sci::col_code(code[j]));
            any |= dbl[i][j];
        }
    if (!any) return;
    uint32_t row[S];
#pragma unroll
    for (int i = 0; i < S; i++) {
        idx[i] = e_idx[g + i];
        grad_offsets(tr, sci::code_x(code[i]), sci::code_y(code[i]), bb_off, row[i], col[i]);
    }
    TC sum[S][S];
#pragma unroll
    for (int v = 0; v < NV; v++) {
        TC c[S];
#pragma unroll
        for (int i = 0; i < S; i++) c[i] = sflip(sci::code_par(code[i]), C[idx[i] * nvec + v0 + v]);
#pragma unroll
        for (int i = 1; i < S; i++) {
            const TC r = scale(conjv(c[i]), wk[v0 + v]);
#pragma unroll
            for (int j = 0; j < i; j++)
                if (dbl[i][j]) {
                    if (v == 0) sum[i][j] = mul(r, c[j]);
                    else mac(sum[i][j], r, c[j]);
                }
        }
    }
#pragma unroll
    for (int i = 1; i < S; i++)
#pragma unroll
        for (int j = 0; j < i; j++)
            if (dbl[i][j]) red(dT + row[i] + col[j], sum[i][j]);
}

// ------------------------------------------------------------------ expansion
// The elements of g1 and g2 from the tables of the three classes.
template <typename TC> struct Tables {
    sci::TabRule tr;
    int norb;
    uint32_t bb_off;
    RefW ref;
    const double *Wt, *D, *DD;
    const TC *A, *Bc, *dT;

    __device__ __forceinline__ double occ_ref(int k) const { return (double)((ref.w[k >> 6] >> (k & 63)) & 1); }
    __device__ __forceinline__ int spin(int p) const { return tr.spinors ? 0 : p >= tr.n; }
    // sum_I w_I n_x n_y
    __device__ __forceinline__ double pair_occ(int x, int y) const
    {
        const double nx = occ_ref(x), ny = occ_ref(y);
        const double dd = x == y ? (nx != 0.0 ? -D[x] : D[x]) : DD[min(x, y) * norb + max(x, y)];
        return *Wt * nx * ny + nx * D[y] + D[x] * ny + dd;
    }
    // <a+_x a_y>, x != y
    __device__ __forceinline__ TC single(int x, int y) const { return add(A[x * norb + y], conjv(A[y * norb + x])); }
    // <a+_x a_y n_k>, x, y and k different
    __device__ __forceinline__ TC spectator(int x, int y, int k) const
    {
        if (spin(x) != spin(y)) return from_real<TC>(0.0);
        const TC b = add(Bc[((int64_t)x * norb + y) * norb + k], conjv(Bc[((int64_t)y * norb + x) * norb + k]));
        return add(scale(single(x, y), occ_ref(k)), b);
    }
    // <a+_p a+_r a_s a_q>
    __device__ __forceinline__ TC two(int p, int q, int r, int s) const
    {
        const TC none = from_real<TC>(0.0);
        if (p == r || q == s) return none;
        if (p == q) return r == s ? from_real<TC>(pair_occ(p, r)) : spectator(r, s, p);
        if (r == s) return spectator(p, q, r);
        if (p == s) return r == q ? from_real<TC>(-pair_occ(p, r)) : neg(spectator(r, q, p));
        if (r == q) return neg(spectator(p, s, r));
        if (spin(p) + spin(r) != spin(q) + spin(s)) return none;
        // a double excitation: both orientations of the pair table
        uint32_t row, col, row2, col2;
        grad_offsets(tr, min(p, r), max(p, r), bb_off, row, col2);
        grad_offsets(tr, min(q, s), max(q, s), bb_off, row2, col);
        const TC u = add(dT[(int64_t)row + col], conjv(dT[(int64_t)row2 + col2]));
        return (p < r) == (q < s) ? u : neg(u);
    }
};

// g1 and, after k_rdm_expand2, the elements of g2 of the other two classes, n^3 of its n^4: a
// thread per (x, y, k), per (x, y) when g2 is null.
template <typename TC> __global__ void k_rdm_expand1(Tables<TC> T, TC *__restrict__ g1, TC *__restrict__ g2)
{
    const int norb = T.norb, kk = g2 ? norb : 1;
    const int64_t n2 = (int64_t)norb * norb, n3 = n2 * norb;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n2 * kk; t += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(t % kk), xy = (int)(t / kk), x = xy / norb, y = xy % norb;
        if (k == 0) g1[xy] = x == y ? from_real<TC>(T.pair_occ(x, x)) : T.single(x, y);
        if (!g2 || x == y) continue;
        if (k == x) {
            const double o = T.pair_occ(x, y);
            g2[x * n3 + x * n2 + y * norb + y] = from_real<TC>(o);      // (x x | y y)
            g2[x * n3 + y * n2 + y * norb + x] = from_real<TC>(-o);     // (x y | y x)
        } else if (k != y && T.spin(x) == T.spin(y)) {
            const TC b = T.spectator(x, y, k);
            g2[x * n3 + y * n2 + k * norb + k] = b;          // (x y | k k)
            g2[k * n3 + k * n2 + x * norb + y] = b;          // (k k | x y)
            g2[x * n3 + k * n2 + k * norb + y] = neg(b);     // (x k | k y)
            g2[k * n3 + y * n2 + x * norb + k] = neg(b);     // (k y | x k)
        }
    }
}

// The double excitations of g2, and zeros elsewhere: every element once in storage order, so that
// g2 needs no clearing.  A CTA takes a (p, q), a warp one row r at a time and its lanes s: what
// belongs to the bra and the spin of s are the warp's, and a row that conserves no spin is only
// stored.  The elements of the other classes are left to k_rdm_expand1: one of them in a warp's
// 32 cost its five to eight FP64 instructions, 16 cycles of the pipe each, as if all were.
// Both kernels at 60 spin-orbitals: 47 us, 118 in one kernel with all classes (a clear and
// scattered stores of all classes took 100); the writes alone, 104 MB, 15 us.
template <typename TC> __global__ void __launch_bounds__(kThreads) k_rdm_expand2(Tables<TC> T, TC *__restrict__ g2)
{
    const int norb = T.norb, n2 = norb * norb;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int pq = blockIdx.x; pq < n2; pq += gridDim.x) {
        const int p = pq / norb, q = pq % norb, ds = T.spin(p) - T.spin(q);
        for (int r = wid; r < norb; r += kThreads / 32) {
            TC *out = g2 + ((int64_t)pq * norb + r) * norb;
            const int ss = ds + T.spin(r);   // the spin of s, by conservation
            const bool any = p != q && p != r && r != q;
            uint32_t row = 0, col2 = 0;
            if (any) grad_offsets(T.tr, min(p, r), max(p, r), T.bb_off, row, col2);
            for (int s = lane; s < norb; s += 32) {
                TC v = from_real<TC>(0.0);
                if (any && s != p && s != q && s != r && T.spin(s) == ss) {
                    uint32_t row2, col;
                    grad_offsets(T.tr, min(q, s), max(q, s), T.bb_off, row2, col);
                    v = add(T.dT[(int64_t)row + col], conjv(T.dT[(int64_t)row2 + col2]));
                    if ((p < r) != (q < s)) v = neg(v);
                }
                out[s] = v;
            }
        }
    }
}

int grid_for(int64_t n)
{
    const int64_t b = (n + kThreads - 1) / kThreads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, sci::kSMs * 16));
}

template <typename TC> struct Walk {
    const TC *C;
    int nvec, v0;
    const double *wk;
    TC *A, *Bc, *dT;  // dT == nullptr: no double-excitation walk
    int CH;
    size_t smem;
    sci::TabRule tr;
    uint32_t bb_off;
};

// the buckets of exactly S members
template <typename TC, int S, int NV> void launch_small(sci_ctx *ctx, const Walk<TC> &w)
{
    const int64_t at = ctx->split2.above[S], n = (ctx->split2.above[S - 1] - at) / S;
    if (n > 0)
        k_rdm_doubles_small<TC, S, NV><<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, ctx->stream>>>(
            ctx->e2_idx + at, ctx->e2_code + at, n, w.tr, w.bb_off, w.C, w.nvec, w.v0, w.wk, w.dT);
}

// the single- and double-excitation walks for one group of NV vectors
template <typename TC, int NV>
int launch_walks(sci_ctx *ctx, const Walk<TC> &w)
{
    if (ctx->e1 > 0) {
        auto ks = ctx->nwords == 4   ? k_rdm_singles<TC, NV, 4>
                  : ctx->nwords == 3 ? k_rdm_singles<TC, NV, 3>
                  : ctx->nwords == 2 ? k_rdm_singles<TC, NV, 2>
                                     : k_rdm_singles<TC, NV, 1>;
        ks<<<grid_for(ctx->e1), kThreads, 0, ctx->stream>>>(ctx->e1_idx, ctx->e1_S, ctx->e1_meta, ctx->e1, ctx->norb,
                                                            ref_words(ctx), w.C, w.nvec, w.v0, w.wk, w.A, w.Bc);
    }
    if (w.dT) {
        const int64_t large = ctx->split2.above[sci::kSortBucket], mid = ctx->split2.above[sci::kSmallBucket];
        if (large > 0) {
            auto kern = k_rdm_doubles<TC, NV>;
            if (w.smem > 32 * 1024 &&
                sci_cuda_check(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w.smem),
                               "rdm12 attr"))
                return SCI_ERR_CUDA;
            kern<<<(unsigned)((large + w.CH - 1) / w.CH), kThreads, w.smem, ctx->stream>>>(
                ctx->e2_idx, ctx->e2_code, ctx->e2_pos, large, w.CH, w.tr, w.bb_off, w.C, w.nvec, w.v0, w.wk, w.dT);
        }
        if (mid > large) {
            auto kern = k_rdm_doubles_sorted<TC, NV>;
            constexpr size_t smem = sort_smem<TC, NV>();
            if (smem > 32 * 1024 &&
                sci_cuda_check(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                               "rdm12 attr"))
                return SCI_ERR_CUDA;
            kern<<<(unsigned)((mid - large + kSortRows - 1) / kSortRows), kThreads, smem, ctx->stream>>>(
                ctx->e2_idx + large, ctx->e2_code + large, ctx->e2_pos + large, mid - large, w.tr, w.bb_off, w.C,
                w.nvec, w.v0, w.wk, w.dT);
        }
        launch_small<TC, 4, NV>(ctx, w);
        launch_small<TC, 3, NV>(ctx, w);
        launch_small<TC, 2, NV>(ctx, w);
    }
    return SCI_OK;
}

// the class tables of a weighted set of vectors, in the context's scratch; with_two: also the
// double-excitation table.  C and the weights are device pointers.
template <typename TC>
int rdm_tables(sci_ctx *ctx, const TC *C, int nvec, const double *wk_dev, bool with_two, Tables<TC> &T)
{
    const int norb = ctx->norb, n = ctx->n;
    const int64_t n2 = (int64_t)norb * norb;
    const int64_t NP = (int64_t)n * (n - 1) / 2;
    const int64_t nT = ctx->spinors ? NP * NP : (int64_t)n * n * n * n + 2 * NP * NP;
    const uint32_t bb_off = ctx->spinors ? 0u : (uint32_t)(NP * NP);
    // scratch: Wt, D[norb], DD[norb^2] (double); A[norb^2], Bc[norb^3], dT[nT] (TC)
    const size_t dbytes = sizeof(double) * (1 + norb + n2);
    const size_t tbytes = sizeof(TC) * (n2 + n2 * norb + (with_two ? nT : 0));
    const size_t need = ((dbytes + 255) & ~(size_t)255) + tbytes;
    if (need > ctx->rdm_bytes) {
        if (ctx->rdm_scratch) cudaFree(ctx->rdm_scratch);
        ctx->rdm_scratch = nullptr, ctx->rdm_bytes = 0;
        if (cudaMalloc(&ctx->rdm_scratch, need) != cudaSuccess) return sci_fail(ctx, SCI_ERR_NOMEM, "rdm12: scratch");
        ctx->rdm_bytes = need;
    }
    unsigned char *base = static_cast<unsigned char *>(ctx->rdm_scratch);
    double *Wt = reinterpret_cast<double *>(base), *D = Wt + 1, *DD = D + norb;
    TC *A = reinterpret_cast<TC *>(base + ((dbytes + 255) & ~(size_t)255));
    TC *Bc = A + n2;
    TC *dT = Bc + n2 * norb;
    if (sci_cuda_check(ctx, cudaMemsetAsync(ctx->rdm_scratch, 0, need, ctx->stream), "rdm12 memset")) return SCI_ERR_CUDA;
    const sci::TabRule tr{ctx->spinors, n};
    // window rows of the large buckets: short windows where there are few (shared memory, and
    // with it the CTAs per SM, is the largest bucket's: 441 members at 30 orbitals;
    // 1.47M entries of buckets above 64: 546 us at 768 rows, 491 at 256)
    const int CH = ctx->split2.above[sci::kSortBucket] / 768 >= sci::kSMs * 16 ? 768 : 256;
    auto stage_bytes = [&](int nv) {
        return (size_t)(CH + ctx->maxb2) * (nv * sizeof(TC) + 2 * sizeof(uint32_t));
    };
    // vectors per walk: at most kMaxVec, fewer when the staged window would not fit
    int kv = kMaxVec;
    while (kv > 1 && stage_bytes(kv) > 200 * 1024) kv >>= 1;
    if (with_two && ctx->e2 > 0 && stage_bytes(kv) > 200 * 1024)
        return sci_fail(ctx, SCI_ERR_OVERFLOW, "rdm12: largest bucket too large for shared memory");
    // the diagonal kernel: DD [norb]^2 and D [norb] in shared memory while they fit (up to
    // 168 orbitals), else accumulated in global memory
    size_t diag_smem = sizeof(double) * ((size_t)norb * norb + norb);
    const bool diag_sm = diag_smem + 4096 <= 227 * 1024;
    auto kd = ctx->nwords == 4   ? (diag_sm ? k_rdm_diag<TC, 4, true> : k_rdm_diag<TC, 4, false>)
              : ctx->nwords == 3 ? (diag_sm ? k_rdm_diag<TC, 3, true> : k_rdm_diag<TC, 3, false>)
              : ctx->nwords == 2 ? k_rdm_diag<TC, 2, true>
                                 : k_rdm_diag<TC, 1, true>;
    if (!diag_sm) diag_smem = 0;
    if (diag_sm && sci_cuda_check(ctx, cudaFuncSetAttribute(kd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                            (int)diag_smem), "rdm12 diag attr"))
        return SCI_ERR_CUDA;
    for (int v0 = 0; v0 < nvec; v0 += kv) {
        const int nv = std::min(kv, nvec - v0);
        kd<<<std::min(grid_for(ctx->M), sci::kSMs * 7), kThreads, diag_smem, ctx->stream>>>(ctx->keys, ctx->M, norb, ref_words(ctx), C, nvec, v0,
                                                                   nv, wk_dev, Wt, D, DD);
        const Walk<TC> wlk{C, nvec, v0, wk_dev, A, Bc, with_two && ctx->e2 > 0 ? dT : nullptr, CH, stage_bytes(nv), tr, bb_off};
        int rc = SCI_OK;
        switch (nv) {
            case 1: rc = launch_walks<TC, 1>(ctx, wlk); break;
            case 2: rc = launch_walks<TC, 2>(ctx, wlk); break;
            case 3: rc = launch_walks<TC, 3>(ctx, wlk); break;
            case 4: rc = launch_walks<TC, 4>(ctx, wlk); break;
            case 5: rc = launch_walks<TC, 5>(ctx, wlk); break;
            case 6: rc = launch_walks<TC, 6>(ctx, wlk); break;
            case 7: rc = launch_walks<TC, 7>(ctx, wlk); break;
            default: rc = launch_walks<TC, 8>(ctx, wlk); break;
        }
        if (rc) return rc;
    }
    T = Tables<TC>{tr, norb, bb_off, ref_words(ctx), Wt, D, DD, A, Bc, dT};
    return SCI_OK;
}

template <typename TC>
int rdm_run(sci_ctx *ctx, const TC *C, int nvec, const double *wk_dev, TC *g1, TC *g2)
{
    Tables<TC> T;
    const int rc = rdm_tables<TC>(ctx, C, nvec, wk_dev, g2 != nullptr, T);
    if (rc) return rc;
    const int n2 = ctx->norb * ctx->norb;
    if (g2) k_rdm_expand2<TC><<<n2, kThreads, 0, ctx->stream>>>(T, g2);
    k_rdm_expand1<TC><<<grid_for((int64_t)n2 * (g2 ? ctx->norb : 1)), kThreads, 0, ctx->stream>>>(T, g1, g2);
    return sci_cuda_check(ctx, cudaGetLastError(), "rdm12 launch") ? SCI_ERR_CUDA : SCI_OK;
}

// the weights of a call (a host array of nvec doubles, NULL = all ones) on the device
int rdm_weights(sci_ctx *ctx, int nvec, const double *weights)
{
    const size_t wbytes = sizeof(double) * nvec;
    if (wbytes > ctx->rdm_wbytes) {
        if (ctx->rdm_w) cudaFree(ctx->rdm_w);
        ctx->rdm_w = nullptr, ctx->rdm_wbytes = 0;
        if (cudaMalloc(&ctx->rdm_w, wbytes) != cudaSuccess) return sci_fail(ctx, SCI_ERR_NOMEM, "rdm12: weights");
        ctx->rdm_wbytes = wbytes;
    }
    std::vector<double> w(nvec, 1.0);
    if (weights) std::copy(weights, weights + nvec, w.begin());
    if (sci_cuda_check(ctx, cudaMemcpyAsync(ctx->rdm_w, w.data(), wbytes, cudaMemcpyHostToDevice, ctx->stream), "rdm12 weights") ||
        sci_cuda_check(ctx, cudaStreamSynchronize(ctx->stream), "rdm12 weights sync"))
        return SCI_ERR_CUDA;
    return SCI_OK;
}

// ------------------------------------------------------------------ gradients of E
// Spin sums of the spin-orbital density matrices (bit p < n alpha p, bit n + p beta p):
//   gamma[p][q]        = sum_s g1[ps][qs]
//   Gamma[p][q][r][s]  = sum_{s1,s2} g2[p s1][q s1][r s2][s s2]
__global__ void k_spin_sum1(int n, Tables<double> T, double *__restrict__ gamma)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * n; t += gridDim.x * blockDim.x) {
        const int p = t / n, q = t % n;
        gamma[t] = p == q ? T.pair_occ(p, p) + T.pair_occ(n + p, n + p) : T.single(p, q) + T.single(n + p, n + q);
    }
}

// straight from the class tables: the spin-orbital g2, sixteen times Gamma, is never formed
__global__ void k_spin_sum2(int n, Tables<double> T, double *__restrict__ Gamma)
{
    const int64_t n4 = (int64_t)n * n * n * n;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x) {
        const int s = (int)(t % n), r = (int)((t / n) % n), q = (int)((t / n / n) % n), p = (int)(t / n / n / n);
        double v = 0.0;
        for (int a = 0; a < 2; a++)
            for (int b = 0; b < 2; b++) v += T.two(p + a * n, q + a * n, r + b * n, s + b * n);
        Gamma[t] = v;
    }
}

// gL[P][i] = sum_k Gamma[i][k] L[P][k] for i, k < n^2 (the chain rule of
// (pq|rs) = sum_P L^P_pq L^P_rs through the free entries of L^P, with Gamma symmetric in
// its two index pairs): an 8 x 32 output tile per CTA, one output per thread, k in steps of 32
// staged in shared memory, the next step's loads in flight meanwhile; FP64 FMA.  The FP64 pipe
// bounds it (2 FMA per clock per SM), so what counts is that every SM has work: 30 orbitals
// and 120 factors are 452 of these tiles, 2.97 per SM.
// Measured: 572 us with 64 x 32 tiles (60 CTAs), 181 us; at the FP64 rate 168 us.
constexpr int kGI = 8, kGP = 32, kGK = 32;
__global__ void __launch_bounds__(256) k_gamma_chol(int nn, int naux, const double *__restrict__ Gamma,
                                                     const double *__restrict__ L, double *__restrict__ gL)
{
    __shared__ double sG[kGI][kGK];
    __shared__ double sL[kGP][kGK + 1];
    const int i0 = blockIdx.x * kGI, P0 = blockIdx.y * kGP;
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    // this thread stages column k0 + tx of row i0 + ty of Gamma and of rows P0 + ty + 8 u of L
    double g, l[4];
    auto load = [&](int k0) {
        const int k = k0 + tx;
        g = i0 + ty < nn && k < nn ? Gamma[(int64_t)(i0 + ty) * nn + k] : 0.0;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int P = P0 + ty + 8 * u;
            l[u] = P < naux && k < nn ? L[(int64_t)P * nn + k] : 0.0;
        }
    };
    double acc = 0.0;
    load(0);
    for (int k0 = 0; k0 < nn; k0 += kGK) {
        __syncthreads();
        sG[ty][tx] = g;
#pragma unroll
        for (int u = 0; u < 4; u++) sL[ty + 8 * u][tx] = l[u];
        __syncthreads();
        if (k0 + kGK < nn) load(k0 + kGK);
#pragma unroll
        for (int kk = 0; kk < kGK; kk++) acc = fma(sG[ty][kk], sL[tx][kk], acc);
    }
    const int P = P0 + tx, i = i0 + ty;
    if (P < naux && i < nn) gL[(int64_t)P * nn + i] = acc;
}

}  // namespace

extern "C" int sci_rdm_grads(sci_ctx *ctx, const double *C, int nvec, const double *weights, double *gamma,
                             double *Gamma, int naux, const double *chol, double *gchol)
{
    if (!ctx) return SCI_ERR_ARG;
    if (!ctx->have_ints || !ctx->have_dets) return sci_fail(ctx, SCI_ERR_STATE, "rdm_grads: integrals and determinants first");
    if (ctx->cplx || ctx->spinors) return sci_fail(ctx, SCI_ERR_ARG, "rdm_grads: real spin-orbital mode only");
    if (nvec < 1 || (ctx->M > 0 && !C)) return sci_fail(ctx, SCI_ERR_ARG, "rdm_grads: need nvec >= 1 and C");
    if ((chol == nullptr) != (gchol == nullptr) || (chol && naux < 1))
        return sci_fail(ctx, SCI_ERR_ARG, "rdm_grads: chol and gchol go together, naux >= 1");
    if (ctx->norb > 256 || ctx->nwords > sci::kMaxWords) return sci_fail(ctx, SCI_ERR_ARG, "rdm_grads: at most 256 orbitals");
    if (sci_cuda_check(ctx, cudaSetDevice(ctx->device), "cudaSetDevice")) return SCI_ERR_CUDA;
    const int n = ctx->n;
    const int64_t nn = (int64_t)n * n, n4 = nn * nn;
    const bool two = Gamma || chol;
    // the spin-summed Gamma, when the caller passes none but needs the contraction
    double *G = Gamma;
    if (two && !Gamma && cudaMalloc(&G, sizeof(double) * n4) != cudaSuccess)
        return sci_fail(ctx, SCI_ERR_NOMEM, "rdm_grads: scratch");
    Tables<double> T;
    int rc = rdm_weights(ctx, nvec, weights);
    if (rc == SCI_OK) rc = rdm_tables<double>(ctx, C, nvec, static_cast<const double *>(ctx->rdm_w), two, T);
    cudaStream_t st = ctx->stream;
    if (rc == SCI_OK && gamma) k_spin_sum1<<<grid_for(nn), kThreads, 0, st>>>(n, T, gamma);
    if (rc == SCI_OK && two) k_spin_sum2<<<grid_for(n4), kThreads, 0, st>>>(n, T, G);
    if (rc == SCI_OK && chol) {
        const dim3 grid((unsigned)((nn + kGI - 1) / kGI), (unsigned)((naux + kGP - 1) / kGP));
        k_gamma_chol<<<grid, 256, 0, st>>>((int)nn, naux, G, chol, gchol);
    }
    if (rc == SCI_OK) rc = sci_cuda_check(ctx, cudaGetLastError(), "rdm_grads launch");
    // Gamma is freed after the queued work has read it
    cudaError_t e = cudaStreamSynchronize(st);
    if (G != Gamma) cudaFree(G);
    if (rc == SCI_OK) rc = sci_cuda_check(ctx, e, "rdm_grads");
    return rc;
}

extern "C" int sci_rdm12(sci_ctx *ctx, const void *C, int nvec, const double *weights, void *rdm1, void *rdm2)
{
    if (!ctx) return SCI_ERR_ARG;
    if (!ctx->have_ints || !ctx->have_dets) return sci_fail(ctx, SCI_ERR_STATE, "rdm12: integrals and determinants first");
    if (nvec < 1 || !rdm1 || (ctx->M > 0 && !C)) return sci_fail(ctx, SCI_ERR_ARG, "rdm12: need nvec >= 1, C and rdm1");
    if (ctx->norb > 256 || ctx->nwords > sci::kMaxWords) return sci_fail(ctx, SCI_ERR_ARG, "rdm12: at most 256 orbitals");
    if (sci_cuda_check(ctx, cudaSetDevice(ctx->device), "cudaSetDevice")) return SCI_ERR_CUDA;
    if (const int rc = rdm_weights(ctx, nvec, weights)) return rc;
    const double *wk = static_cast<const double *>(ctx->rdm_w);
    if (ctx->cplx)
        return rdm_run<zdbl>(ctx, static_cast<const zdbl *>(C), nvec, wk, static_cast<zdbl *>(rdm1), static_cast<zdbl *>(rdm2));
    return rdm_run<double>(ctx, static_cast<const double *>(C), nvec, wk, static_cast<double *>(rdm1), static_cast<double *>(rdm2));
}
