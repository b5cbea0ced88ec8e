// Panel factorisation of the blocked LU (Algorithm 1's batched LU, P A = L U
// with partial pivoting) and the inverses of its diagonal blocks.
//
// A panel is the columns [k, k + nb) of rows [k, n) of one box.  A cluster of
// C CTAs (256 threads each) takes one box; row r belongs for the whole panel
// to thread r mod 256 of CTA (r / 256) mod C, and rows never move while the
// panel is factored.  The panel goes left to right in blocks of IB columns
// that a thread holds for its RPT rows in registers:
//   1. load the block; for each earlier block: the rows that were its pivots
//      hand their entries over, the block's unit triangle (its inverse, kept)
//      turns them into rows of U, and every other row subtracts its stored
//      multipliers times them (16 multiply-adds per value read back);
//   2. factor the block: per column every warp offers its largest candidate
//      with its row, the CTA picks one after one barrier (in a cluster the
//      CTAs' offers are exchanged through distributed shared memory and a
//      cluster barrier), and every thread eliminates with the winning row
//      from shared memory;
//   3. multipliers of the rows still active go back to the matrix.
// At the end the first CTA places the pivot rows on top, moves the rows they
// displaced and writes the step's permutation (perm[r]: the old row at
// position r, as a sequence of row swaps would give it).
//
// What bounds it: with many boxes the multiply-adds of the elimination
// (R nb^2 / 2 per box: the FP32 pipes at 128 a clock, the FP64 pipes at 2);
// with few, the chain of nb pivots, about 500 clocks each with one CTA and
// 1100 with a cluster, and the elimination divided by C.  Keeping rows in
// registers leaves one shared-memory read of the pivot row per RPT rows where
// a panel in shared memory took two reads and a write per multiply-add.
#include <algorithm>
#include <climits>

#include "hps_internal.h"
#include "hps_ptx.cuh"

namespace hps {

namespace {

constexpr int PT = 256, PW = PT / 32;   // threads and warps of a panel CTA
constexpr int kMaxCluster = 8;

__device__ __forceinline__ unsigned cluster_size()
{
    unsigned v;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(v));
    return v;
}
__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned v;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
    return v;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t remote_addr(const void* p, unsigned rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void remote_store(uint32_t a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, unsigned long long v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, int v)
{
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Pivot key of a value: larger for larger magnitudes, 1 for a NaN (taken only
// when nothing else is left); 0 is kept for rows that are no candidates.
__device__ __forceinline__ unsigned long long pivot_key(float x)
{
    return x != x ? 1ull : (unsigned long long)(__float_as_uint(x) & 0x7FFFFFFFu) + 2ull;
}
__device__ __forceinline__ unsigned long long pivot_key(double x)
{
    return x != x ? 1ull : ((unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull) + 2ull;
}

// Largest key over the lanes and, among its holders, the lowest row; true on
// the lane that holds it.  FP32 keys fit 32 bits.
template <typename T>
__device__ __forceinline__ bool warp_argmax(unsigned long long& key, int& row)
{
    bool mine = key != 0;
    if constexpr (sizeof(T) == 4) {
        const unsigned k = (unsigned)key, m = __reduce_max_sync(0xffffffffu, k);
        mine = mine && k == m;
        key = m;
    } else {
        const unsigned h = (unsigned)(key >> 32), mh = __reduce_max_sync(0xffffffffu, h);
        const unsigned l = h == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, l);
        mine = mine && h == mh && l == ml;
        key = ((unsigned long long)mh << 32) | ml;
    }
    const int r = __reduce_min_sync(0xffffffffu, mine ? row : INT_MAX);
    mine = mine && row == r;
    row = r;
    return mine;
}

template <typename T, int N>
__device__ __forceinline__ void load_row(T (&d)[N], const T* s)   // 16-byte aligned
{
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int per = 16 / sizeof(T);
#pragma unroll
    for (int i = 0; i < N / per; ++i) {
        const V v = reinterpret_cast<const V*>(s)[i];
        const T* e = reinterpret_cast<const T*>(&v);
#pragma unroll
        for (int u = 0; u < per; ++u) d[per * i + u] = e[u];
    }
}
template <typename T, int N>
__device__ __forceinline__ void store_row(T* s, const T (&d)[N])
{
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int per = 16 / sizeof(T);
#pragma unroll
    for (int i = 0; i < N / per; ++i) {
        V v;
        T* e = reinterpret_cast<T*>(&v);
#pragma unroll
        for (int u = 0; u < per; ++u) e[u] = d[per * i + u];
        reinterpret_cast<V*>(s)[i] = v;
    }
}

template <typename T>
struct PanelArgs {
    T* M;
    long long ldm, sM;
    int n, k, nb;
    int* perm;
    long long sP;
    int* status;
    const int* skip;
};

// Shared memory of a panel CTA.
template <typename T, int IB>
struct PanelSmem {
    alignas(16) T inv[kMaxNB / IB][IB][IB];        // inverses of the blocks' unit lower triangles
    alignas(16) T raw[2][IB][IB], u[IB][IB];       // a block's pivot rows before (alternating: a CTA may run one
                                                   // block ahead of its cluster) and after its triangle
    alignas(16) T cand[2][PW][IB];                 // the warps' offers
    alignas(16) T offer[2][kMaxCluster][IB];       // the CTAs' offers
    unsigned long long ckey[2][PW], okey[2][kMaxCluster];
    int crow[2][PW], orow[2][kMaxCluster];
    int prow[kMaxNB];                              // row chosen for each column
    int pp[kMaxNB];                                // position it had been swapped to
    int moved_from[kMaxNB], moved_to[kMaxNB], nmoved;
    unsigned char is_pivot[kMaxNB];
    int sing;
};

// CTAs per SM: two of FP32 (77 KiB of shared memory at nb = 128), three of FP64 where a row is 32 registers.
template <typename T>
constexpr int panel_min_blocks(int regs) { return regs <= 32 && sizeof(T) == 8 ? 3 : regs <= 64 ? 2 : 1; }

template <typename T, int RPT, int IB>
__global__ void __launch_bounds__(PT, panel_min_blocks<T>(RPT * IB * (int)sizeof(T) / 4))
k_panel(const PanelArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PanelSmem<T, IB>& s = *reinterpret_cast<PanelSmem<T, IB>*>(smem_raw);
    constexpr size_t kHead = (sizeof(PanelSmem<T, IB>) + 15) / 16 * 16;
    const int nb = a.nb, nblk = (nb + IB - 1) / IB, ldl = nblk * IB;
    T* LU = reinterpret_cast<T*>(smem_raw + kHead);   // [ldl][ldl]: pivot rows (unit L below, U on and above)
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int box = blockIdx.x / C;
    if (a.skip && a.skip[box]) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R0 = a.n - a.k;
    T* P = a.M + box * a.sM + (long long)a.k * a.ldm + a.k;   // the panel's corner
    auto row_of = [&](int rr) { return (rr * C + rank) * PT + tid; };

    int pidx[RPT];   // column whose pivot the row became; -1 active, -2 no such row
#pragma unroll
    for (int rr = 0; rr < RPT; ++rr) pidx[rr] = row_of(rr) < R0 ? -1 : -2;
    if (tid < kMaxNB) s.is_pivot[tid] = 0;
    if (tid == 0) { s.sing = 0; s.nmoved = 0; }
    if (C > 1) cluster_sync();   // every CTA of the cluster runs before its shared memory is written

    T x[RPT][IB];
    for (int b = 0; b < nblk; ++b) {
        const int jb = b * IB, w = min(IB, nb - jb);
        // 1. the block's entries, brought up to date
#pragma unroll
        for (int rr = 0; rr < RPT; ++rr) {
#pragma unroll
            for (int c = 0; c < IB; ++c) x[rr][c] = T(0);
            if (pidx[rr] != -2) {
                const T* src = P + (long long)row_of(rr) * a.ldm + jb;
                if (w == IB) load_row<T, IB>(x[rr], src);
                else {
#pragma unroll
                    for (int c = 0; c < IB; ++c)
                        if (c < w) x[rr][c] = src[c];
                }
            }
        }
        for (int e = 0; e < b; ++e) {
            const int je = e * IB;
#pragma unroll
            for (int rr = 0; rr < RPT; ++rr)
                if (pidx[rr] >= je && pidx[rr] < je + IB) {
                    if (C == 1) store_row<T, IB>(s.raw[e & 1][pidx[rr] - je], x[rr]);
                    else
                        for (int d = 0; d < C; ++d) {
                            const uint32_t to = remote_addr(s.raw[e & 1][pidx[rr] - je], (unsigned)d);
#pragma unroll
                            for (int c = 0; c < IB; ++c) remote_store(to + c * (uint32_t)sizeof(T), x[rr][c]);
                        }
                }
            if (C == 1) __syncthreads();
            else cluster_sync();
            if (tid < IB * IB) {
                const int i = tid / IB, c = tid - i * IB;
                T acc0 = T(0), acc1 = T(0);
#pragma unroll
                for (int t = 0; t < IB; t += 2) {   // the inverse is zero above its diagonal
                    acc0 += s.inv[e][i][t] * s.raw[e & 1][t][c];
                    acc1 += s.inv[e][i][t + 1] * s.raw[e & 1][t + 1][c];
                }
                const T v = acc0 + acc1;
                s.u[i][c] = v;
                LU[(je + i) * ldl + jb + c] = v;
            }
            __syncthreads();
            constexpr int JC = 16 / sizeof(T);   // multipliers read at a time (16 bytes)
#pragma unroll 1
            for (int j0 = 0; j0 < IB; j0 += JC) {
                T l[RPT][JC];
#pragma unroll
                for (int rr = 0; rr < RPT; ++rr) {
                    const bool on = pidx[rr] == -1 || pidx[rr] >= je + IB;
#pragma unroll
                    for (int j = 0; j < JC; ++j) l[rr][j] = T(0);
                    if (on) load_row<T, JC>(l[rr], P + (long long)row_of(rr) * a.ldm + je + j0);
                }
#pragma unroll
                for (int j = 0; j < JC; ++j) {
                    T uv[IB];
                    load_row<T, IB>(uv, s.u[j0 + j]);
#pragma unroll
                    for (int rr = 0; rr < RPT; ++rr)
#pragma unroll
                        for (int c = 0; c < IB; ++c) x[rr][c] -= l[rr][j] * uv[c];
                }
            }
        }
        // 2. factor the block
#pragma unroll
        for (int c = 0; c < IB; ++c) {
            if (c < w) {
                const int cur = c & 1;
                unsigned long long key = 0;
                int row = INT_MAX, brr = 0;
#pragma unroll
                for (int rr = 0; rr < RPT; ++rr) {
                    const unsigned long long kk = pidx[rr] == -1 ? pivot_key(x[rr][c]) : 0ull;
                    if (kk > key) { key = kk; row = row_of(rr); brr = rr; }
                }
                const bool mine = warp_argmax<T>(key, row);
                if (mine) {
#pragma unroll
                    for (int rr = 0; rr < RPT; ++rr)
                        if (rr == brr) store_row<T, IB>(s.cand[cur][warp], x[rr]);
                }
                if (lane == 0) { s.ckey[cur][warp] = key; s.crow[cur][warp] = row; }
                __syncthreads();
                // the CTA's best (every warp finds it for itself)
                key = lane < PW ? s.ckey[cur][lane] : 0ull;
                row = lane < PW ? s.crow[cur][lane] : INT_MAX;
                const unsigned who = __ballot_sync(0xffffffffu, warp_argmax<T>(key, row));
                int best = who ? __ffs((int)who) - 1 : 0;
                const T* pv = s.cand[cur][best];
                if (C > 1) {
                    if (warp == 0) {
                        for (int e = lane; e < C * IB; e += 32) {
                            const int d = e / IB, cc = e - d * IB;
                            remote_store(remote_addr(&s.offer[cur][rank][cc], (unsigned)d), pv[cc]);
                        }
                        if (lane < C) {
                            remote_store(remote_addr(&s.okey[cur][rank], (unsigned)lane), key);
                            remote_store(remote_addr(&s.orow[cur][rank], (unsigned)lane), row);
                        }
                    }
                    cluster_sync();
                    key = lane < C ? s.okey[cur][lane] : 0ull;
                    row = lane < C ? s.orow[cur][lane] : INT_MAX;
                    const unsigned whoc = __ballot_sync(0xffffffffu, warp_argmax<T>(key, row));
                    best = whoc ? __ffs((int)whoc) - 1 : 0;
                    pv = s.offer[cur][best];
                }
                T p[IB];
                load_row<T, IB>(p, pv);
                T piv = p[c];
                if (piv == T(0)) {   // exactly singular: record it and keep the arithmetic finite
                    if (tid == 0) s.sing = 1;
                    piv = T(1);
                }
                const T rinv = T(1) / piv;
                if (tid < IB) LU[(jb + c) * ldl + jb + tid] = pv[tid];
                if (tid == 32) {
                    s.prow[jb + c] = row;
                    if (row < nb) s.is_pivot[row] = 1;
                    int pos = row;   // follow the swaps that moved the row before
                    while (pos < jb + c) pos = s.pp[pos];
                    s.pp[jb + c] = pos;
                }
#pragma unroll
                for (int rr = 0; rr < RPT; ++rr) {
                    if (row_of(rr) == row) pidx[rr] = jb + c;
                    if (pidx[rr] == -1) {
                        const T l = x[rr][c] * rinv;
                        x[rr][c] = l;
#pragma unroll
                        for (int cc = c + 1; cc < IB; ++cc) x[rr][cc] -= l * p[cc];
                    }
                }
            }
        }
        // 3. multipliers of the active rows
#pragma unroll
        for (int rr = 0; rr < RPT; ++rr)
            if (pidx[rr] == -1) {
                T* dst = P + (long long)row_of(rr) * a.ldm + jb;
                if (w == IB) store_row<T, IB>(dst, x[rr]);
                else {
#pragma unroll
                    for (int c = 0; c < IB; ++c)
                        if (c < w) dst[c] = x[rr][c];
                }
            }
        __syncthreads();
        // the block's unit triangle inverted: a column per lane, each entry
        // taken off the later ones as soon as it is known
        if (b + 1 < nblk && tid < IB) {
            T y[IB];
#pragma unroll
            for (int i = 0; i < IB; ++i) y[i] = i == tid ? T(1) : T(0);
#pragma unroll
            for (int t = 0; t < IB; ++t)
#pragma unroll
                for (int i = t + 1; i < IB; ++i) y[i] -= LU[(jb + i) * ldl + jb + t] * y[t];
#pragma unroll
            for (int i = 0; i < IB; ++i) s.inv[b][i][tid] = y[i];
        }
        __syncthreads();
    }
    __threadfence();
    if (C > 1) cluster_sync();   // every row's multipliers are in memory; no distributed access follows
    else __syncthreads();
    if (rank != 0) return;

    // Pivot rows' multipliers of earlier blocks into LU, and where the rows
    // that they displaced from the top go: a row swapped to a position that a
    // later column takes moves on with it.
    for (int idx = tid; idx < nb * ldl; idx += PT) {
        const int j = idx / ldl, c = idx - j * ldl;
        if (c < j / IB * IB) LU[idx] = __ldcg(P + (long long)s.prow[j] * a.ldm + c);
    }
    if (tid < nb && !s.is_pivot[tid]) {
        int pos = tid;
        while (pos < nb) pos = s.pp[pos];
        const int q = atomicAdd(&s.nmoved, 1);
        s.moved_from[q] = tid;
        s.moved_to[q] = pos;
    }
    int* pb = a.perm + box * a.sP;
    for (int r = tid; r < R0; r += PT) pb[r] = r < nb ? s.prow[r] : r;
    __syncthreads();
    for (int idx = tid; idx < s.nmoved * nb; idx += PT) {
        const int q = idx / nb, c = idx - q * nb;
        P[(long long)s.moved_to[q] * a.ldm + c] = __ldcg(P + (long long)s.moved_from[q] * a.ldm + c);
    }
    if (tid < s.nmoved) pb[s.moved_to[tid]] = s.moved_from[tid];
    __syncthreads();
    for (int idx = tid; idx < nb * nb; idx += PT) {
        const int j = idx / nb, c = idx - j * nb;
        P[(long long)j * a.ldm + c] = LU[j * ldl + c];
    }
    if (tid == 0 && s.sing && a.status[box] == 0) a.status[box] = HPS_ESINGULAR;
}

// ---------------------------------------------------------------- diagonal inverses

constexpr int TI = 512;   // threads of an inverse

// Inverse of a triangle held in A (P x P, row-major, P a power of two >= 16,
// padded with the identity): the unit lower triangle below A's diagonal
// (lower) or the upper triangle with its diagonal.  The 16 x 16 diagonal
// blocks are inverted by substitution (a column per thread), then blocks of
// doubling size b are joined: for [[A1, 0], [C, D]] the off-diagonal block
// of the inverse is -D^{-1} (C A1^{-1}); for [[A1, B], [0, D]] it is
// -A1^{-1} (B D^{-1}).  The middle product is parked in the free triangle of
// A.  X must be zero on entry and receives the inverse.  A zero diagonal
// entry is read as 1 (the box is already flagged singular).
template <typename T>
__device__ void tri_inverse(T* A, T* X, int P, bool lower, int tid)
{
    if (tid < P) {
        const int q0 = (tid >> 4) << 4, c = tid - q0;
        T y[16], d[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            y[i] = i == c ? T(1) : T(0);
            const T v = A[(q0 + i) * P + q0 + i];
            d[i] = lower ? T(1) : T(1) / (v == T(0) ? T(1) : v);
        }
        if (lower) {
#pragma unroll
            for (int t = 0; t < 16; ++t)
#pragma unroll
                for (int i = t + 1; i < 16; ++i) y[i] -= A[(q0 + i) * P + q0 + t] * y[t];
        } else {
#pragma unroll
            for (int t = 15; t >= 0; --t) {
                y[t] *= d[t];
#pragma unroll
                for (int i = 0; i < t; ++i) y[i] -= A[(q0 + i) * P + q0 + t] * y[t];
            }
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) X[(q0 + i) * P + q0 + c] = y[i];
    }
    __syncthreads();
    for (int b = 16; b < P; b *= 2) {
        const int items = (P / (2 * b)) * b * b;
        // middle products into the free triangle of A
        for (int it = tid; it < items; it += TI) {
            const int pr = it / (b * b), e = it - pr * b * b, r = e / b, c = e - r * b, i0 = 2 * b * pr;
            T acc = T(0);
            if (lower) {   // C A1^{-1}: C = A[i0+b+r][i0+t], A1^{-1} lower
                for (int t = c; t < b; ++t) acc += A[(i0 + b + r) * P + i0 + t] * X[(i0 + t) * P + i0 + c];
                A[(i0 + r) * P + i0 + b + c] = acc;
            } else {       // B D^{-1}: B = A[i0+r][i0+b+t], D^{-1} upper
                for (int t = 0; t <= c; ++t) acc += A[(i0 + r) * P + i0 + b + t] * X[(i0 + b + t) * P + i0 + b + c];
                A[(i0 + b + r) * P + i0 + c] = acc;
            }
        }
        __syncthreads();
        for (int it = tid; it < items; it += TI) {
            const int pr = it / (b * b), e = it - pr * b * b, r = e / b, c = e - r * b, i0 = 2 * b * pr;
            T acc = T(0);
            if (lower) {   // -D^{-1} (C A1^{-1}), D^{-1} lower
                for (int t = 0; t <= r; ++t) acc -= X[(i0 + b + r) * P + i0 + b + t] * A[(i0 + t) * P + i0 + b + c];
                X[(i0 + b + r) * P + i0 + c] = acc;
            } else {       // -A1^{-1} (B D^{-1}), A1^{-1} upper
                for (int t = r; t < b; ++t) acc -= X[(i0 + r) * P + i0 + t] * A[(i0 + b + t) * P + i0 + c];
                X[(i0 + r) * P + i0 + b + c] = acc;
            }
        }
        __syncthreads();
    }
}

// F top = -L11^{-1} (blockIdx.x = 0) and B top = -U11^{-1} (1) of each box's
// factored diagonal block.  One CTA each, so that the two run side by side.
template <typename T>
__global__ void __launch_bounds__(TI)
k_tri_inv(const T* __restrict__ M, long long ldm, long long sM, int k, int nb, T* __restrict__ Ftop, long long ldf,
          long long sF, T* __restrict__ Btop, long long ldb, long long sB, const int* skip)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int box = blockIdx.y, tid = threadIdx.x;
    const bool lower = blockIdx.x == 0;
    if (skip && skip[box]) return;
    int Pd = 16;
    while (Pd < nb) Pd *= 2;
    T* A = reinterpret_cast<T*>(smem_raw);   // Pd x Pd, padded with the identity
    T* X = A + Pd * Pd;
    const T* D = M + box * sM + (long long)k * ldm + k;
    for (int idx = tid; idx < Pd * Pd; idx += TI) {
        const int r = idx / Pd, c = idx - r * Pd;
        const bool in = r < nb && c < nb && (lower ? c < r : c >= r);
        A[idx] = in ? D[(long long)r * ldm + c] : (!lower && r == c ? T(1) : T(0));
        X[idx] = T(0);
    }
    __syncthreads();
    tri_inverse<T>(A, X, Pd, lower, tid);
    T* out = lower ? Ftop + box * sF : Btop + box * sB;
    const long long ldo = lower ? ldf : ldb;
    for (int idx = tid; idx < nb * nb; idx += TI) {
        const int r = idx / nb, c = idx - r * nb;
        out[r * ldo + c] = -X[r * Pd + c];
    }
}

template <typename T>
using PanelKernel = void (*)(const PanelArgs<T>);

struct PanelShape {
    int rpt, ib;
    int occ;   // CTAs per SM
};

template <typename T>
PanelKernel<T> panel_kernel(int i);
template <>
PanelKernel<float> panel_kernel<float>(int i)
{
    switch (i) {
        case 0: return k_panel<float, 1, 16>;
        case 1: return k_panel<float, 2, 16>;
        case 2: return k_panel<float, 4, 16>;
        default: return k_panel<float, 8, 16>;
    }
}
template <>
PanelKernel<double> panel_kernel<double>(int i)
{
    switch (i) {
        case 0: return k_panel<double, 1, 16>;
        case 1: return k_panel<double, 2, 16>;
        case 2: return k_panel<double, 4, 16>;
        default: return k_panel<double, 8, 8>;
    }
}
template <typename T>
PanelShape panel_shape(int i)
{
    static const PanelShape f[4] = {{1, 16, 2}, {2, 16, 2}, {4, 16, 2}, {8, 16, 1}};
    static const PanelShape d[4] = {{1, 16, 3}, {2, 16, 2}, {4, 16, 1}, {8, 8, 1}};
    return sizeof(T) == 4 ? f[i] : d[i];
}
template <typename T>
size_t panel_smem(int ib, int nb)
{
    const size_t head = ib == 16 ? sizeof(PanelSmem<T, 16>) : sizeof(PanelSmem<T, 8>), ldl = align_up((size_t)nb, (size_t)ib);
    return align_up(head, 16) + ldl * ldl * sizeof(T);
}

}  // namespace

template <typename T>
void launch_panel(T* M, long long ldm, long long sM, int n, int k, int nb, int* perm, long long sP, T* Ftop,
                  long long ldf, long long sF, T* Btop, long long ldb, long long sB, int* status, const int* skip,
                  int nbox, cudaStream_t st)
{
    static const bool once = [] {
        for (int i = 0; i < 4; ++i)
            cudaFuncSetAttribute(panel_kernel<T>(i), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)panel_smem<T>(panel_shape<T>(i).ib, sizeof(T) == 4 ? kMaxNB : 64));
        cudaFuncSetAttribute(k_tri_inv<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(2 * (sizeof(T) == 4 ? kMaxNB * kMaxNB : 64 * 64) * sizeof(T)));
        return true;
    }();
    (void)once;
    // Rows per thread and cluster size: the fewest waves of (chain of nb pivots
    // + the elimination's issue), with the measured clocks of one pivot: about
    // 500 alone, 1100 in a cluster, and per row of a thread 160 (FP32) or 5200
    // (FP64) shared by the CTAs of an SM.
    const int R0 = n - k;
    int bi = 3, bc = kMaxCluster;
    double best = -1.0;
    for (int i = 0; i < 4; ++i) {
        const PanelShape sh = panel_shape<T>(i);
        for (int c = 1; c <= kMaxCluster; c *= 2) {
            if ((long long)PT * sh.rpt * c < R0) continue;
            // blocks of 8 columns only for FP64 panels that nothing else holds, so that
            // the arithmetic does not depend on the batch
            if (sh.ib != 16 && R0 <= PT * 4 * kMaxCluster) continue;
            const long long ctas = (long long)nbox * c, slots = 152LL * sh.occ;
            const double waves = (double)((ctas + slots - 1) / slots);
            const double share = (double)std::min<long long>(sh.occ, (ctas + 151) / 152);
            const double rows = (double)std::min((long long)sh.rpt, ((long long)R0 + PT * c - 1) / (PT * c));
            const double cost = waves * ((c == 1 ? 500.0 : 1100.0) + share * rows * (sizeof(T) == 4 ? 160.0 : 5200.0));
            if (best < 0 || cost < best) { best = cost; bi = i; bc = c; }
        }
    }
    PanelArgs<T> a{M, ldm, sM, n, k, nb, perm, sP, status, skip};
    prof_begin(KC_PANEL, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nbox * bc));
    cfg.blockDim = dim3(PT);
    cfg.dynamicSmemBytes = panel_smem<T>(panel_shape<T>(bi).ib, nb);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)bc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, panel_kernel<T>(bi), a);
    int Pd = 16;
    while (Pd < nb) Pd *= 2;
    k_tri_inv<T><<<dim3(2, (unsigned)nbox), TI, 2 * (size_t)Pd * Pd * sizeof(T), st>>>(M, ldm, sM, k, nb, Ftop, ldf, sF,
                                                                                       Btop, ldb, sB, skip);
    prof_end(KC_PANEL, st, (double)nbox * R0 * (double)nb * nb, (double)nbox * 2.0 * R0 * nb * sizeof(T));
}

template void launch_panel<float>(float*, long long, long long, int, int, int, int*, long long, float*, long long,
                                  long long, float*, long long, long long, int*, const int*, int, cudaStream_t);
template void launch_panel<double>(double*, long long, long long, int, int, int, int*, long long, double*, long long,
                                   long long, double*, long long, long long, int*, const int*, int, cudaStream_t);

}  // namespace hps
