// Panel factorisation of the blocked LU (Algorithm 1's batched LU, P A = L U
// with partial pivoting) and the inverses of its diagonal blocks.
//
// A panel is the columns [k, k + nb) of rows [k, n) of one box.  A cluster of
// C CTAs (256 threads each) takes one box, groups of 32 rows dealt out to the
// CTAs and then to their warps; a row belongs to one thread for the whole
// panel, and rows never move while it is factored.  The panel goes left to right in blocks of IB columns
// that a thread holds for its RPT rows in registers:
//   1. load the block; for each earlier block: the rows that were its pivots
//      hand their entries over, the block's unit triangle (its inverse, kept)
//      turns them into rows of U, and every other row subtracts its stored
//      multipliers times them (16 multiply-adds per value read back; FP64 as
//      digit products on the tensor cores, see hps_digits.cuh, except in boxes
//      whose scales lie too far apart for them);
//   2. factor the block: per column every warp offers its largest candidate
//      with its row, the CTA picks one after one barrier (in a cluster the
//      CTAs' offers are exchanged through distributed shared memory and a
//      cluster barrier), and every thread eliminates with the winning row
//      from shared memory;
//   3. multipliers of the rows still active go to a scratch block by columns,
//      where a warp reads and writes whole lines.
// At the end every row goes to its place in the matrix: pivot rows on top, rows
// they displaced to the places that they left; perm[r] is the old row at
// position r.
//
// What bounds it: the chain of nb pivots with one box per CTA and SM (a barrier,
// the comparison of eight offers and the first of the next column's entries per
// pivot; a cluster adds its barrier, 390 clocks, and the exchange), and with many
// boxes the issue of the elimination, R nb^2 / 2 multiply-adds.  Keeping rows in
// registers leaves one shared-memory read of the pivot row per RPT rows where a
// panel in shared memory took two reads and a write per multiply-add.  Against
// that form: 128 columns of 1000 rows 475 -> 217 us (one box) and 1.94 -> 0.92 ms
// (512 boxes); 64 FP64 columns of 216 rows 660 -> 160 us.
#include <algorithm>
#include <atomic>
#include <climits>
#include <type_traits>

#include "hps_digits.cuh"
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
__device__ __forceinline__ void remote_store(uint32_t a, unsigned v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, int v)
{
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Pivot key of a value: larger for larger magnitudes, 1 for a NaN (taken only
// when nothing else is left); 0 is kept for rows that are no candidates.
template <typename T>
using PivotKey = typename std::conditional<sizeof(T) == 4, unsigned, unsigned long long>::type;
__device__ __forceinline__ unsigned pivot_key(float x)
{
    return x != x ? 1u : (__float_as_uint(x) & 0x7FFFFFFFu) + 2u;
}
__device__ __forceinline__ unsigned long long pivot_key(double x)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
    return u > 0x7FF0000000000000ull ? 1ull : u + 2ull;
}

// Largest key over the lanes and, among its holders, the lowest row; true on
// the lane that holds it.
__device__ __forceinline__ bool warp_argmax(unsigned& key, int& row)
{
    const unsigned m = __reduce_max_sync(0xffffffffu, key);
    bool mine = key != 0 && key == m;
    key = m;
    const int r = __reduce_min_sync(0xffffffffu, mine ? row : INT_MAX);
    mine = mine && row == r;
    row = r;
    return mine;
}
__device__ __forceinline__ bool warp_argmax(unsigned long long& key, int& row)
{
    const unsigned h = (unsigned)(key >> 32), mh = __reduce_max_sync(0xffffffffu, h);
    const unsigned l = h == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, l);
    bool mine = key != 0 && h == mh && l == ml;
    key = ((unsigned long long)mh << 32) | ml;
    const int r = __reduce_min_sync(0xffffffffu, mine ? row : INT_MAX);
    mine = mine && row == r;
    row = r;
    return mine;
}

// Index of the best of eight offers (keys and rows on 16 bytes), with its key
// and row: a tree of comparisons, the reduction instructions' latency saved.
template <typename K>
__device__ __forceinline__ int best_offer(const K* ks, const int* rs, K& key, int& row)
{
    K k[8];
    int r[8], id[8];
#pragma unroll
    for (int i = 0; i < 8 * (int)sizeof(K) / 16; ++i)
        *reinterpret_cast<uint4*>(&k[i * 16 / (int)sizeof(K)]) = reinterpret_cast<const uint4*>(ks)[i];
#pragma unroll
    for (int i = 0; i < 2; ++i) *reinterpret_cast<int4*>(&r[4 * i]) = reinterpret_cast<const int4*>(rs)[i];
#pragma unroll
    for (int i = 0; i < 8; ++i) id[i] = i;
#pragma unroll
    for (int h = 4; h > 0; h >>= 1)
#pragma unroll
        for (int i = 0; i < h; ++i)
            if (k[i + h] > k[i] || (k[i + h] == k[i] && r[i + h] < r[i])) {
                k[i] = k[i + h];
                r[i] = r[i + h];
                id[i] = id[i + h];
            }
    key = k[0];
    row = r[0];
    return id[0];
}

// 1 / x.  FP64: on the integer pipe (a division is ten dependent operations of
// 64 clocks a warp on the FP64 pipe): y, 1 / m to 22 bits from FP32, then
// y (1 + e + e^2) with e = 1 - m y in fixed point, |e|^3 below 2^-66, rounded
// once; below 0.51 units in the last place.
__device__ __forceinline__ float reciprocal(float x) { return 1.0f / x; }
__device__ __forceinline__ double reciprocal(double x)
{
    const uint64_t u = (uint64_t)__double_as_longlong(x);
    const int ex = (int)(u >> 52) & 0x7ff;
    if (ex - 1 > 2042) return 1.0 / x;   // subnormal results, infinities, NaN
    if (ex == 0) return 1.0 / x;
    const uint64_t M = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;             // m 2^52
    const float mf = __uint_as_float(0x3F800000u | (uint32_t)((M >> 29) & 0x7FFFFFu));
    const uint32_t yb = __float_as_uint(__frcp_rn(mf));
    const uint32_t Y = yb >= 0x3F800000u ? 0x80000000u : ((yb & 0x7FFFFFu) | 0x800000u) << 7;   // y 2^31
    const long long E = -(long long)(M * (uint64_t)Y);                               // e 2^83 (2^83 = 0 mod 2^64)
    const long long t = __mul64hi(E, (long long)((uint64_t)Y << 12));                // y e 2^62
    const long long R = (long long)((uint64_t)Y << 31) + t + (__mul64hi(t, E) >> 19);
    const uint64_t mant = (uint64_t)(R + 256) >> 9;
    return __longlong_as_double((long long)((u & 0x8000000000000000ull) | (((uint64_t)(2044 - ex) << 52) + mant)));
}

// a -= l u over a row; FP32 two entries an instruction (the same rounding).
template <int N>
__device__ __forceinline__ void sub_row(float (&a)[N], float l, const float (&u)[N])
{
    const float m = -l;
#pragma unroll
    for (int i = 0; i < N; i += 2)
        asm("{\n\t.reg .b64 x, y, z;\n\t"
            "mov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %2};\n\tmov.b64 z, {%3, %4};\n\t"
            "fma.rn.f32x2 x, y, z, x;\n\t"
            "mov.b64 {%0, %1}, x;\n\t}"
            : "+f"(a[i]), "+f"(a[i + 1])
            : "f"(m), "f"(u[i]), "f"(u[i + 1]));
}
template <int N>
__device__ __forceinline__ void sub_row(double (&a)[N], double l, const double (&u)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) a[i] -= l * u[i];
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

// 16-byte unit q of row r in a warp's tile of 32 rows of 64 bytes, swizzled so
// that neither a lane per row nor four lanes per row meet in a bank.
template <typename T>
__device__ __forceinline__ float4* tile_unit(T* tile, int r, int q)
{
    return reinterpret_cast<float4*>(tile) + r * 4 + (q ^ ((r >> 1) & 3));
}

// The same for rows of 128 bytes (16 FP64 values).
__device__ __forceinline__ double2* tile_unit128(double* tile, int r, int q)
{
    return reinterpret_cast<double2*>(tile) + r * 8 + (q ^ (r & 7));
}

// D += A B, m16n8k16, FP16 in, FP32 accumulate.
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}

template <typename T>
struct PanelArgs {
    T* M;
    long long ldm, sM;
    int n, k, nb;
    T* Lt;           // scratch [nb][n - k] per box: the multipliers by columns while the panel is factored
    long long sL;
    int* perm;
    long long sP;
    int* status;
    const int* skip;
    int* wide;       // FP64: boxes that run on plain sums (is_wide; written by the panel at k = 0)
    int axis, dims;
};

// FP64 LUs run from exact digits (hps_digit.cu), which are as good as FP64 sums
// relative to the largest entries of a row and a column of a product.  A matrix
// whose scales lie far apart needs its small entries too, and its LU runs on
// plain sums: true where the rows' largest entries lie 2^9 or more apart, or (axis,
// dims: a collocation matrix of axis^dims nodes) where the second differences of
// its axes do by more than 2^12.  Errors of S against long double, from digits :
// on FP64 sums (geometric means of norms over ten 2-D boxes, p = 16): rows 2^5
// apart (every smooth or rough problem; at most 2^7 at p <= 24) 1 : 1.3, 2^13
// (coefficients that jump by 1e8 from node to node) 1.2 : 1, 2^19 to 2^33 (1e10 to
// 1e14) 19 to 26 : 1, 2^39 (1e16) 1500 : 1; impedance leaves of side 1 / 64, 2^10
// apart before their rows were scaled, 15 : 1.  Boxes of sides 1 : 100 keep the norm
// but lose a digit of the median entry, 1 : 1e6 all but two of the small ones.
//
// A row's scale is the exponent of its largest entry within two columns of the
// diagonal, where collocation, impedance and interface matrices have entries of
// that size (all of M would take 0.7 ms to read of the 101 of 512 boxes at p =
// 12); rows with nothing beside it, the identity that pads a separator to its
// level's size, have none.  The axes are compared along the grid's diagonal, where the neighbours on
// every axis have the same 1-D index; half of these nodes decide.  Every CTA of the
// first panel finds the same answer for itself: a kernel for it took 5 of the 117
// us of one box at p = 5.
__device__ __noinline__ bool is_wide(const double* __restrict__ A, long long ldm, int n, int axis, int dims)
{
    __shared__ int top[2], flat;   // largest exponent, 2047 less the smallest; nodes with axes far apart
    if (threadIdx.x == 0) top[0] = top[1] = flat = 0;
    __syncthreads();
    auto expo = [&](long long r, long long c) { return ((unsigned)__double2hiint(A[r * ldm + c]) & 0x7FFFFFFFu) >> 20; };
    int hi = 0, lo = 0;
    for (int r = threadIdx.x; r < n; r += PT) {
        unsigned beside = 0;
#pragma unroll
        for (int u = -2; u <= 2; ++u)
            if (u != 0 && r + u >= 0 && r + u < n) beside = max(beside, expo(r, r + u));
        const int t = (int)max(beside, expo(r, r));
        if (beside) {
            hi = max(hi, t);
            lo = max(lo, 2047 - t);
        }
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_max_sync(0xffffffffu, lo);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&top[0], hi);
        atomicMax(&top[1], lo);
    }
    if (dims && (int)threadIdx.x + 1 < axis) {
        const long long node = 1 + axis + (dims == 3 ? (long long)axis * axis : 0), r = threadIdx.x * node;
        const unsigned x = expo(r, r + 1), y = expo(r, r + axis), z = dims == 3 ? expo(r, r + (long long)axis * axis) : x;
        if (max(max(x, y), z) > min(min(x, y), z) + 12) atomicAdd(&flat, 1);
    }
    __syncthreads();
    return top[0] + top[1] >= 2047 + 9 || (dims && 2 * flat >= axis - 1 && flat > 0);
}

// Entry (row, column) of the product of an earlier block's multipliers with u as
// an FP64 sum; l, u: the first multiplier and value, a step apart each.
template <int IB>
__device__ __noinline__ double plain_entry(const double* l, long long step, const double* u)
{
    double s = 0.0;
    for (int k = 0; k < IB; ++k) s = fma(l[k * step], u[k * IB], s);
    return s;
}

// Shared memory of a panel CTA.
template <typename T, int IB>
struct PanelSmem {
    // per warp: 32 rows of 64 bytes between row and column order (FP64: of IB values, for its products)
    alignas(16) T tile[PW][sizeof(T) == 8 ? 32 * IB : 512];
    alignas(16) T inv[kMaxNB / IB][IB][IB];        // inverses of the blocks' unit lower triangles
    alignas(16) T raw[2][IB][IB], u[IB][IB];       // a block's pivot rows before (alternating: a CTA may run one
                                                   // block ahead of its cluster) and after its triangle
    alignas(16) uint2 ud[sizeof(T) == 8 ? IB / 8 : 1][DG_S][32];   // FP64: u's digits as MMA operands
    int ue[IB];                                    // and the scales of its columns
    alignas(16) T cand[2][PW][IB];                 // the warps' offers
    alignas(16) T offer[2][kMaxCluster][IB];       // the CTAs' offers
    T crcp[2][PW], orcp[2][kMaxCluster];           // reciprocals of the offered pivots
    alignas(16) PivotKey<T> ckey[2][PW];
    alignas(16) PivotKey<T> okey[2][kMaxCluster];
    alignas(16) int crow[2][PW];
    alignas(16) int orow[2][kMaxCluster];
    int prow[kMaxNB];                              // row chosen for each column
    int vac[kMaxNB], dest[kMaxNB];                 // places left by pivots below the top; where displaced rows go
    int nd[4], nv[4];
    unsigned char is_pivot[kMaxNB];
    int sing;
};
static_assert(PW == 8 && kMaxCluster == 8, "best_offer compares eight");
static_assert(PT * 8 * kMaxCluster == kPanelMaxRows, "the largest shape below");

// CTAs per SM by the registers of a thread's rows: two of up to 64 (FP32) or 32 (FP64, whose products take 90 more).
template <typename T>
constexpr int panel_min_blocks(int regs) { return regs <= (sizeof(T) == 4 ? 64 : 32) ? 2 : 1; }

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
    bool hard = false;   // FP64: left products as plain sums
    if constexpr (sizeof(T) == 8) hard = a.k == 0 ? is_wide(P, a.ldm, a.n, a.axis, a.dims) : a.wide[box] != 0;
    auto row_of = [&](int rr) { return ((rr * PW + warp) * C + rank) * 32 + lane; };
    // the warp's row groups that exist (all of a group's lanes may still be past the last row)
    const int nrr = min(RPT, max(0, ((R0 + 31) / 32 - rank - warp * C + PW * C - 1) / (PW * C)));

    int pidx[RPT];   // column whose pivot the row became; -1 active, -2 no such row
#pragma unroll
    for (int rr = 0; rr < RPT; ++rr) pidx[rr] = row_of(rr) < R0 ? -1 : -2;
    if (tid < kMaxNB) s.is_pivot[tid] = 0;
    if (tid == 0) s.sing = 0;
    if (tid < 2 * kMaxCluster) (&s.okey[0][0])[tid] = 0;
    if (C > 1) cluster_sync();   // every CTA of the cluster runs before its shared memory is written

    constexpr int CU = 16 / sizeof(T), CW = 4 * CU;   // entries of a 16-byte unit and of a 64-byte row piece
    T* tile = s.tile[warp];
    auto tile_row = [](T* t, int r, int q) {   // FP64 product rows: IB values each
        if constexpr (IB == 16) return tile_unit128(reinterpret_cast<double*>(t), r, q);
        else return reinterpret_cast<double2*>(tile_unit(t, r, q));
    };
    T* Lt = a.Lt + box * a.sL;
    T x[RPT][IB];
    for (int b = 0; b < nblk; ++b) {
        const int jb = b * IB, w = min(IB, nb - jb);
        // 1. the block's entries, brought up to date.  Rows are read 64 bytes at a
        // time by four lanes each (a lane per row would touch 32 lines an
        // instruction) and turned through the warp's tile.
#pragma unroll
        for (int rr = 0; rr < RPT; ++rr) {
#pragma unroll
            for (int c = 0; c < IB; ++c) x[rr][c] = T(0);
            if (rr >= nrr) continue;
            const int row0 = row_of(rr) - lane;
            if (w == IB) {
#pragma unroll
                for (int h = 0; h < IB / CW; ++h) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = 8 * i + (lane >> 2);
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (row0 + r < R0)
                            v = *reinterpret_cast<const float4*>(P + (long long)(row0 + r) * a.ldm + jb + h * CW + (lane & 3) * CU);
                        *tile_unit(tile, r, lane & 3) = v;
                    }
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 v = *tile_unit(tile, lane, q);
                        const T* e = reinterpret_cast<const T*>(&v);
#pragma unroll
                        for (int t = 0; t < CU; ++t) x[rr][h * CW + q * CU + t] = e[t];
                    }
                    __syncwarp();
                }
            } else if (pidx[rr] != -2) {
                const T* src = P + (long long)row_of(rr) * a.ldm + jb;
#pragma unroll
                for (int c = 0; c < IB; ++c)
                    if (c < w) x[rr][c] = src[c];
            }
        }
        for (int e = 0; e < b; ++e) {
            const int je = e * IB;
            // FP32: multipliers read ahead per row, the first ones before the barrier
            constexpr int JC = sizeof(T) == 8 ? 1 : 16 / RPT;
            T l[RPT][JC];
            auto load_l = [&](int j0) {
#pragma unroll
                for (int rr = 0; rr < RPT; ++rr) {
                    const bool on = pidx[rr] == -1 || pidx[rr] >= je + IB;
#pragma unroll
                    for (int j = 0; j < JC; ++j) l[rr][j] = on ? Lt[(long long)(je + j0 + j) * R0 + row_of(rr)] : T(0);
                }
            };
            if constexpr (sizeof(T) == 4) load_l(0);
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
            if constexpr (sizeof(T) == 4) {
#pragma unroll 1
                for (int j0 = 0; j0 < IB; j0 += JC) {
                    T lc[RPT][JC];
#pragma unroll
                    for (int rr = 0; rr < RPT; ++rr)
#pragma unroll
                        for (int j = 0; j < JC; ++j) lc[rr][j] = l[rr][j];
                    if (j0 + JC < IB) load_l(j0 + JC);
#pragma unroll
                    for (int j = 0; j < JC; ++j) {
                        T uv[IB];
                        load_row<T, IB>(uv, s.u[j0 + j]);
#pragma unroll
                        for (int rr = 0; rr < RPT; ++rr)
                            if (rr < nrr) sub_row(x[rr], lc[rr][j], uv);
                    }
                }
            } else {
                // FP64: the product of the multipliers with u from exact digits
                // (K = IB <= 16: every accumulator stays below 2^21); as 16 multiply-adds
                // per entry on the FP64 pipe, 64 clocks a warp each, it took seven times as long
                const int g = lane >> 2, q = lane & 3;
                if (warp < IB / 8) {
                    double v[4];
                    int ex = E_MIN;
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int kk = 2 * q + (t & 1) + 8 * (t >> 1);
                        v[t] = kk < IB ? s.u[kk < IB ? kk : 0][8 * warp + g] : 0.0;
                        ex = max(ex, exp_of(v[t]));
                    }
                    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 1));
                    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 2));
                    uint32_t d[DG_S][2];
                    split4(v, ex, d);
#pragma unroll
                    for (int t = 0; t < DG_S; ++t) s.ud[warp][t][lane] = make_uint2(d[t][0], d[t][1]);
                    if (q == 0) s.ue[8 * warp + g] = ex == E_BAD ? E_NAN : ex - 1018;
                }
                __syncthreads();
#pragma unroll
                for (int rr = 0; rr < RPT; ++rr) {
                    if (rr >= nrr) continue;
                    const bool mineon = pidx[rr] == -1 || pidx[rr] >= je + IB;
                    const uint32_t onm = __ballot_sync(0xffffffffu, mineon);
                    const int row0 = row_of(rr) - lane;
#pragma unroll 1
                    for (int mt = 0; mt < 2; ++mt) {
                        uint32_t ad[2][DG_S][2];
                        int ea[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int rl = 16 * mt + 8 * h + g;
                            const bool on = onm >> rl & 1;
                            double v[4];
                            int ex = E_MIN;
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                const int kk = 2 * q + (t & 1) + 8 * (t >> 1);
                                v[t] = on && kk < IB ? Lt[(long long)(je + kk) * R0 + row0 + rl] : 0.0;
                                ex = max(ex, exp_of(v[t]));
                            }
                            ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 1));
                            ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 2));
                            split4(v, ex, ad[h]);
                            ea[h] = ex == E_BAD || hard ? E_NAN : ex;   // E_NAN: every entry of the row a plain sum
                        }
#pragma unroll 1
                        for (int nt = 0; nt < IB / 8; ++nt) {
                            uint2 bd[DG_S];
#pragma unroll
                            for (int t = 0; t < DG_S; ++t) bd[t] = s.ud[nt][t][lane];
                            // accumulators two at a time, joined as they are done
                            long long V[4] = {0, 0, 0, 0};
#pragma unroll
                            for (int t = 0; t < DG_S; t += 2) {
                                float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                                for (int i = 0; i <= t; ++i)
                                    mma16816(c0, ad[0][i][0], ad[1][i][0], ad[0][i][1], ad[1][i][1], bd[t - i]);
#pragma unroll
                                for (int i = 0; i <= t + 1; ++i)
                                    mma16816(c1, ad[0][i][0], ad[1][i][0], ad[0][i][1], ad[1][i][1], bd[t + 1 - i]);
                                constexpr float MG = 12582912.0f;
                                constexpr uint32_t MB = 0x4B400000u;
#pragma unroll
                                for (int o = 0; o < 4; ++o) {
                                    const int w2 = (int)(__float_as_uint(__fadd_rn(c0[o], MG)) * 256u +
                                                         (__float_as_uint(__fadd_rn(c1[o], MG)) - MB * 257u));
                                    if (t == 0) V[o] = (long long)((uint64_t)(uint32_t)(w2 << 7) << 32);
                                    else if (t == 2) V[o] += (long long)w2 * (1 << 23);
                                    else if (t == 4) V[o] += (long long)w2 * 128;
                                    else V[o] += (w2 + 256) >> 9;
                                }
                            }
                            const int2 ue = *reinterpret_cast<const int2*>(&s.ue[8 * nt + 2 * q]);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                int eb0, eb1;
                                double2 r;
                                r.x = round_fixed(V[2 * h], ea[h] + ue.x, eb0);
                                r.y = round_fixed(V[2 * h + 1], ea[h] + ue.y, eb1);
                                if (((unsigned)eb0 > 2045u || (unsigned)eb1 > 2045u) && (onm >> (16 * mt + 8 * h + g) & 1)) {
                                    const double* l = Lt + (long long)je * R0 + row0 + 16 * mt + 8 * h + g;
                                    if ((unsigned)eb0 > 2045u) r.x = plain_entry<IB>(l, R0, &s.u[0][8 * nt + 2 * q]);
                                    if ((unsigned)eb1 > 2045u) r.y = plain_entry<IB>(l, R0, &s.u[0][8 * nt + 2 * q + 1]);
                                }
                                *tile_row(tile, 16 * mt + 8 * h + g, 4 * nt + q) = r;
                            }
                        }
                    }
                    __syncwarp();
                    if (mineon) {
#pragma unroll
                        for (int c = 0; c < IB / 2; ++c) {
                            const double2 r = *tile_row(tile, lane, c);
                            x[rr][2 * c] -= r.x;
                            x[rr][2 * c + 1] -= r.y;
                        }
                    }
                    __syncwarp();
                }
            }
        }
        // 2. factor the block.  A row's entries move one register down per
        // column, so that the column at hand is always x[.][0] and the loop stays
        // small (unrolled over the columns it outgrows the instruction cache);
        // the multipliers fill the registers that come free at the end.
        PivotKey<T> key;
        int row, brr;
        T rcp;
        bool mine;
        // the warp's offer for the column in x[.][0], with the reciprocal that its
        // elimination will need taken while the reductions run
        auto offer = [&]() {
            key = 0;
            row = INT_MAX;
            brr = 0;
            T xb = T(1);
#pragma unroll
            for (int rr = 0; rr < RPT; ++rr) {
                const PivotKey<T> kk = pidx[rr] == -1 ? pivot_key(x[rr][0]) : PivotKey<T>(0);
                if (kk > key) { key = kk; row = row_of(rr); brr = rr; xb = x[rr][0]; }
            }
            rcp = reciprocal(xb == T(0) ? T(1) : xb);   // a zero pivot: recorded below, the arithmetic stays finite
            mine = warp_argmax(key, row);
        };
        offer();
#pragma unroll 1
        for (int c = 0; c < w; ++c) {
            const int cur = c & 1;
            if (mine) {
#pragma unroll
                for (int rr = 0; rr < RPT; ++rr)
                    if (rr == brr) store_row<T, IB>(s.cand[cur][warp], x[rr]);
                s.crcp[cur][warp] = rcp;
            }
            if (lane == 0) { s.ckey[cur][warp] = key; s.crow[cur][warp] = row; }
            __syncthreads();
            int best = best_offer(s.ckey[cur], s.crow[cur], key, row);
            const T* pv = s.cand[cur][best];
            T rinv = s.crcp[cur][best];
            if (C > 1) {
                if (warp == 0) {
                    for (int e = lane; e < C * IB; e += 32) {
                        const int d = e / IB, cc = e - d * IB;
                        remote_store(remote_addr(&s.offer[cur][rank][cc], (unsigned)d), pv[cc]);
                    }
                    if (lane < C) {
                        remote_store(remote_addr(&s.okey[cur][rank], (unsigned)lane), key);
                        remote_store(remote_addr(&s.orow[cur][rank], (unsigned)lane), row);
                        remote_store(remote_addr(&s.orcp[cur][rank], (unsigned)lane), rinv);
                    }
                }
                cluster_sync();
                best = best_offer(s.okey[cur], s.orow[cur], key, row);
                pv = s.offer[cur][best];
                rinv = s.orcp[cur][best];
            }
            if (tid < IB) LU[(jb + c) * ldl + jb + ((tid + c) & (IB - 1))] = pv[tid];
            if (tid == 32) {
                s.prow[jb + c] = row;
                if (row < nb) s.is_pivot[row] = 1;
                if (key == 2) s.sing = 1;   // |pivot| = 0
            }
            T l[RPT];
#pragma unroll
            for (int rr = 0; rr < RPT; ++rr) {
                if (row_of(rr) == row) pidx[rr] = jb + c;
                l[rr] = x[rr][0] * rinv;
            }
            constexpr int PC = 16 / sizeof(T);   // pivot-row entries read at a time (16 bytes)
#pragma unroll
            for (int i0 = 0; i0 < IB; i0 += PC) {
                T p[PC];
                load_row<T, PC>(p, pv + i0);
#pragma unroll
                for (int u = 0; u < PC; ++u) {
                    const int i = i0 + u;
                    if (i == 0) continue;
                    // entries past the block's columns are multipliers: left as they are
                    const bool col = i < IB - c;
                    const T pu = col ? p[u] : T(0);
#pragma unroll
                    for (int rr = 0; rr < RPT; ++rr)
                        if (rr < nrr) {
                            if constexpr (sizeof(T) == 4) x[rr][i - 1] = x[rr][i] - l[rr] * pu;
                            else x[rr][i - 1] = col ? x[rr][i] - l[rr] * pu : x[rr][i];
                        }
                    if (i == 1) offer();   // the next column is known first; its reductions overlap the rest
                }
            }
#pragma unroll
            for (int rr = 0; rr < RPT; ++rr) x[rr][IB - 1] = l[rr];
        }
        for (int c = w; c < IB; ++c) {   // a ragged block: turn the multipliers to the front
#pragma unroll
            for (int rr = 0; rr < RPT; ++rr) {
                const T l = x[rr][0];
#pragma unroll
                for (int i = 1; i < IB; ++i) x[rr][i - 1] = x[rr][i];
                x[rr][IB - 1] = l;
            }
        }
        // 3. multipliers of the active rows, by columns
#pragma unroll
        for (int rr = 0; rr < RPT; ++rr)
            if (pidx[rr] == -1) {
#pragma unroll
                for (int c = 0; c < IB; ++c)
                    if (c < w) Lt[(long long)(jb + c) * R0 + row_of(rr)] = x[rr][c];
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
    if (C > 1) cluster_sync();   // every row's multipliers are in memory; no distributed access follows
    else __syncthreads();

    // Every row that became no pivot goes to its place: below the panel's top
    // it stays; the i-th row that pivots displaced from the top takes the i-th
    // place that they left below it.
    {
        const bool disp = tid < nb && !s.is_pivot[tid < nb ? tid : 0], left = tid < nb && s.prow[tid < nb ? tid : 0] >= nb;
        const uint32_t md = __ballot_sync(0xffffffffu, disp), mv = __ballot_sync(0xffffffffu, left);
        const uint32_t below = (1u << lane) - 1;
        if (lane == 0 && warp < 4) { s.nd[warp] = __popc(md); s.nv[warp] = __popc(mv); }
        __syncthreads();
        int od = __popc(md & below), ov = __popc(mv & below);
        for (int q = 0; q < warp && q < 4; ++q) { od += s.nd[q]; ov += s.nv[q]; }
        if (left) s.vac[ov] = s.prow[tid];
        __syncthreads();
        if (disp) s.dest[tid] = s.vac[od];
        __syncthreads();
    }
    int* pb = a.perm + box * a.sP;
    for (int rr = 0; rr < nrr; ++rr) {
        const int row = row_of(rr);
        int pos = -1;
        if (row < R0 && (row >= nb || !s.is_pivot[row])) {
            bool pivot = false;
            if (row >= nb) {
#pragma unroll
                for (int q = 0; q < RPT; ++q)
                    if (q == rr) pivot = pidx[q] >= 0;
            }
            if (!pivot) {
                pos = row < nb ? s.dest[row] : row;
                pb[pos] = row;
            }
        }
        for (int c0 = 0; c0 < nb; c0 += CW) {
            if (c0 + CW <= nb) {
                __syncwarp();
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float4 v;
                    T* e = reinterpret_cast<T*>(&v);
#pragma unroll
                    for (int t = 0; t < CU; ++t) e[t] = pos >= 0 ? Lt[(long long)(c0 + q * CU + t) * R0 + row] : T(0);
                    *tile_unit(tile, lane, q) = v;
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = 8 * i + (lane >> 2), to = __shfl_sync(0xffffffffu, pos, r);
                    if (to >= 0)
                        *reinterpret_cast<float4*>(P + (long long)to * a.ldm + c0 + (lane & 3) * CU) =
                            *tile_unit(tile, r, lane & 3);
                }
            } else if (pos >= 0) {
                for (int c = c0; c < nb; ++c) P[(long long)pos * a.ldm + c] = Lt[(long long)c * R0 + row];
            }
        }
    }
    if (rank != 0) return;
    if constexpr (sizeof(T) == 8)
        if (tid == 0 && a.k == 0) a.wide[box] = hard;

    // The pivot rows on top: their multipliers of earlier blocks join what LU holds.
    for (int idx = tid; idx < nb * ldl; idx += PT) {
        const int j = idx % nb, c = idx / nb;
        if (c < j / IB * IB) LU[j * ldl + c] = __ldcg(Lt + (long long)c * R0 + s.prow[j]);
    }
    if (tid < nb) pb[tid] = s.prow[tid];
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
    // V neighbouring columns per item: one 16-byte read and one broadcast per V
    // multiply-adds (X is zero on the far side of its diagonal, so a loop may
    // start or end at the item's first or last column)
    constexpr int V = 16 / sizeof(T);
    for (int b = 16; b < P; b *= 2) {
        const int items = (P / (2 * b)) * b * (b / V);
        // middle products into the free triangle of A
        for (int it = tid; it < items; it += TI) {
            const int pr = it / (b * (b / V)), e = it - pr * (b * (b / V)), r = e / (b / V), c = (e - r * (b / V)) * V,
                      i0 = 2 * b * pr;
            T acc[V] = {};
            const T* m = lower ? A + (i0 + b + r) * P + i0 : A + (i0 + r) * P + i0 + b;
            const T* xr = lower ? X + i0 * P + i0 + c : X + (i0 + b) * P + i0 + b + c;
            const int t0 = lower ? c : 0, t1 = lower ? b : c + V;   // C A1^{-1} (A1^{-1} lower) or B D^{-1} (upper)
#pragma unroll 4
            for (int t = t0; t < t1; ++t) {
                T xv[V];
                load_row<T, V>(xv, xr + t * P);
#pragma unroll
                for (int q = 0; q < V; ++q) acc[q] += m[t] * xv[q];
            }
            store_row<T, V>(lower ? A + (i0 + r) * P + i0 + b + c : A + (i0 + b + r) * P + i0 + c, acc);
        }
        __syncthreads();
        for (int it = tid; it < items; it += TI) {
            const int pr = it / (b * (b / V)), e = it - pr * (b * (b / V)), r = e / (b / V), c = (e - r * (b / V)) * V,
                      i0 = 2 * b * pr;
            T acc[V] = {};
            const T* m = lower ? X + (i0 + b + r) * P + i0 + b : X + (i0 + r) * P + i0;
            const T* xr = lower ? A + i0 * P + i0 + b + c : A + (i0 + b) * P + i0 + c;
            const int t0 = lower ? 0 : r, t1 = lower ? r + 1 : b;   // -D^{-1} (..), D^{-1} lower, or -A1^{-1} (..), upper
#pragma unroll 4
            for (int t = t0; t < t1; ++t) {
                T xv[V];
                load_row<T, V>(xv, xr + t * P);
#pragma unroll
                for (int q = 0; q < V; ++q) acc[q] -= m[t] * xv[q];
            }
            store_row<T, V>(lower ? X + (i0 + b + r) * P + i0 + c : X + (i0 + r) * P + i0 + b + c, acc);
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
#pragma unroll 8
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
    int occ;        // CTAs per SM
    double group;   // clocks of a pivot per group of 32 rows of an SM's CTAs
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
    static const PanelShape f[4] = {{1, 16, 2, 100}, {2, 16, 2, 100}, {4, 16, 2, 100}, {8, 16, 1, 125}};
    static const PanelShape d[4] = {{1, 16, 2, 190}, {2, 16, 1, 240}, {4, 16, 1, 330}, {8, 8, 1, 380}};
    return sizeof(T) == 4 ? f[i] : d[i];
}
template <typename T>
size_t panel_smem(int ib, int nb)
{
    const size_t head = ib == 16 ? sizeof(PanelSmem<T, 16>) : sizeof(PanelSmem<T, 8>), ldl = align_up((size_t)nb, (size_t)ib);
    return align_up(head, 16) + ldl * ldl * sizeof(T);
}


// Shared-memory limits of the kernels, a property of a kernel on a device: raised
// when a device runs its first panel.
template <typename T>
void panel_attributes()
{
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_relaxed) & bit) return;
    const int nb = sizeof(T) == 4 ? kMaxNB : 64;
    for (int i = 0; i < 4; ++i)
        cudaFuncSetAttribute(panel_kernel<T>(i), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)panel_smem<T>(panel_shape<T>(i).ib, nb));
    cudaFuncSetAttribute(k_tri_inv<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * nb * nb * (int)sizeof(T));
    done.fetch_or(bit, std::memory_order_relaxed);
}

__global__ void k_refuse(int nbox, int* status)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nbox && status[b] == 0) status[b] = HPS_EINVAL;
}

}  // namespace

template <typename T>
void launch_panel(T* M, long long ldm, long long sM, int n, int k, int nb, int* perm, long long sP, T* Ftop,
                  long long ldf, long long sF, T* Btop, long long ldb, long long sB, int* status, const int* skip,
                  int* wide, int axis, int dims, int nbox, cudaStream_t st)
{
    panel_attributes<T>();
    // Rows per thread and cluster size: the fewest waves of (chain of a pivot +
    // the elimination's issue), in clocks fitted to timings of every shape at 1
    // to 512 boxes and 64 to 5832 rows: the chain takes about 1500 alone and 2900
    // in a cluster for FP32, 4300 and 6000 for FP64 (barriers, the offer, the
    // left products' latency, spread over the pivots), and a group of 32 rows what
    // panel_shape lists.  FP32, 128 columns: one box of 1000 rows 217 to 254 us
    // by shape, 512 boxes of 2744 rows 3.6 ms with four CTAs of four rows a thread
    // against 3.9 with two of eight; FP64, 64 columns: 8 boxes of 216 rows 160 us
    // with one CTA a box against 204 with eight.
    const int R0 = n - k, sms = sm_count();
    if (R0 > kPanelMaxRows) {   // every caller's matrices are smaller (static_assert): nothing is left out silently
        k_refuse<<<(unsigned)((nbox + 255) / 256), 256, 0, st>>>(nbox, status);
        return;
    }
    int bi = 3, bc = kMaxCluster;
    double best = -1.0;
    for (int i = 0; i < 4; ++i) {
        const PanelShape sh = panel_shape<T>(i);
        for (int c = 1; c <= kMaxCluster; c *= 2) {
            if ((long long)PT * sh.rpt * c < R0) continue;
            // blocks of 8 columns only for FP64 panels that nothing else holds, so that
            // the arithmetic does not depend on the batch
            if (sh.ib != 16 && R0 <= PT * 4 * kMaxCluster) continue;
            const long long ctas = (long long)nbox * c, slots = (long long)sms * sh.occ;
            const double waves = (double)((ctas + slots - 1) / slots);
            const double share = (double)std::min<long long>(sh.occ, (ctas + sms - 1) / sms);
            const double groups = (double)((R0 + 32 * c - 1) / (32 * c));
            const double chain = sizeof(T) == 4 ? (c == 1 ? 1500.0 : 2900.0) : (c == 1 ? 4300.0 : 6000.0);
            const double cost = waves * (chain + share * groups * sh.group) + 0.2 * c;
            if (best < 0 || cost < best) { best = cost; bi = i; bc = c; }
        }
    }
    // Rows are read and written 16 bytes at a time: M is 256-byte aligned, ldm a
    // multiple of 8 and k one of 16 (make_plan rounds every stride up, steps are
    // NB wide).  The multipliers' scratch is the step's F block, which the inverse and the
    // product after this overwrite
    PanelArgs<T> a{M, ldm, sM, n, k, nb, Ftop, sF, perm, sP, status, skip, wide, axis, dims};
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
                                  long long, float*, long long, long long, int*, const int*, int*, int, int, int, cudaStream_t);
template void launch_panel<double>(double*, long long, long long, int, int, int, int*, long long, double*, long long,
                                   long long, double*, long long, long long, int*, const int*, int*, int, int, int, cudaStream_t);

}  // namespace hps
