// FP64 products on the tensor cores from exact 8-bit digits (sm_103a, tcgen05).
//
// The FP64 pipes of this part do 2 multiply-adds per clock and SM, its FP16
// tensor cores 4096, so the FP64 path's products O <- src + alpha A B run as
// sums of exact integer products (the splitting idea of Ozaki, Ogita, Oishi
// and Rump, Numer. Algorithms 59, 2012):
//
//   * every row of A and every column of B gets a power-of-two scale from its
//     largest exponent over the K <= 64 indices of a product, and each entry
//     becomes a 62-bit fixed-point number under that scale (the entry's 53
//     significant bits are kept whole down to 2^-9 of the row's maximum, the
//     absolute cut is 2^-62 of it), written as eight balanced base-256 digits
//     (the leading one at most 64);
//   * a digit is an FP16 integer of magnitude <= 128, so digit products and
//     their sums over K and over all pairs (i, j) with i + j = t stay below
//     8 * 64 * 2^14 = 2^23 and are exact in the FP32 accumulators;
//   * the accumulators t = 0..7 (36 of the 64 digit pairs; the rest adds up to
//     about 2^-59 of the product of the two scales, 2^-53 if all its digits
//     were largest and of one sign) are joined in 64-bit integers with a unit
//     of 2^-57, rounded once to FP64 and added to the source.
//
// So the only roundings are those three; a plain FP64 sum rounds K times, but
// relative to its own terms, not to the scales: operands whose scales say little
// about an entry are summed plainly on the FP64 pipe (CHECK below; is_wide in hps_panel.cu).
// Against a higher-precision solve, the LU built on these products is as close
// as or closer than the one on FP64 multiply-adds (tests/test_gpu_digit.py).
// Results outside the normal range, and all of a row or column that holds an
// infinity or a NaN, are summed as they stand on the FP64 pipe instead.
//
// Layout.  One CTA of 512 threads per SM takes a 128-row strip of A (split
// once, 128 KiB of digits in shared memory) across a range of column tiles of
// 32.  Per tile all threads split the 64 x 32 block of B (double buffered), one
// thread issues 32 MMAs (A digit i against the stacked digits 0..7-i of B, N =
// 32 (8 - i): the diagonals t land in consecutive TMEM columns), and while they
// run every warp joins 32 x 8 outputs of the tile before (TMEM holds two tiles
// of 8 x 32 columns, all 512).
//
// What bounds it, measured at M x N x K = 1000 x 1536 x 64 and 160 products
// (18 TFLOP/s, 8800 clocks a tile; the FP64 pipes' 1.1): the warps of a CTA pass
// through the phases of a tile together, so their times add up: joining 2000
// clocks, splitting 1000, waiting for the MMAs 700 (2300 by themselves), the
// adds to O 1800, and 3000 for barriers, TMEM and shared-memory traffic.  Groups
// of warps on alternate tiles, a tile's MMAs issued by the last warp to arrive
// or by a warp of their own were each slower (2.0, 2.4 and 2.6 ms against 1.74):
// they cost registers or coalesced reads of B, and the MMAs' latency shows.
// Whole calls: 512 boxes at p = 12 (DtN, particular and reconstruction) 1001 ->
// 101 ms, cross-term leaves 225 -> 39 to 41 ms.
#include <algorithm>

#include "hps_digits.cuh"
#include "hps_internal.h"
#include "hps_ptx.cuh"

namespace hps {

namespace {

constexpr int DG_BM = 128, DG_BN = 32, DG_K = 64;      // tile
constexpr int DG_THREADS = 512, DG_WARPS = DG_THREADS / 32;
constexpr uint32_t A_PLANE = DG_BM * 128;              // one digit of A: rows of 64 FP16 (128 B, 128B swizzle)
constexpr uint32_t B_PLANE = DG_BN * 128;
constexpr uint32_t B_BUF = DG_S * B_PLANE;
constexpr uint32_t STAGE = 32 * 8 * 8;                 // per warp: 32 x 8 results
constexpr uint32_t OFF_B = DG_S * A_PLANE, OFF_ST = OFF_B + 2 * B_BUF;
constexpr size_t DG_SMEM = OFF_ST + DG_WARPS * STAGE + 1024;
constexpr uint64_t DG_WAIT_NS = 2000000000ull;

struct DgArgs {
    GemmArgs<double> g;
    int tiles_n, per;   // column tiles, and how many of them a CTA takes
    int reach;          // CHECK: an entry's large factors are those within 2^-reach of their scales
};

// Sum of acc_t 2^(45 - 8 t) (unit 2^-57 of the scales' product 2^(E - 1016 ..))
// rounded once to FP64.  The accumulators are turned to integers by adding
// 1.5 2^23 (the conversion instruction runs at 16 lanes a clock and took 93 %
// of the kernel's time): exact below 2^22, which holds for t <= 4 (the leading
// digits are at most 64).  t = 5 is first cut to a multiple of 4, whose rest
// joins t = 6, 7; those only need to be right to a fraction of the unit, so
// their sum is taken in FP32 (an error below 2^-4 units).
__device__ __forceinline__ double join(const float (&a)[DG_S], int E, int& eb_out)
{
    constexpr float MG = 12582912.0f;   // 1.5 2^23, bits 0x4B400000
    constexpr uint32_t MB = 0x4B400000u;
    auto bits = [](float x) { return __float_as_uint(x); };
    const float h = __fmaf_rn(a[5], 0.25f, MG);
    const float r5 = __fmaf_rn(-4.0f, __fsub_rn(h, MG), a[5]);                        // -2 .. 2
    const float lo = __fmaf_rn(r5, 256.0f, __fmaf_rn(a[7], 0.00390625f, a[6]));       // unit 2^-3
    const int low = (int)(bits(__fmaf_rn(lo, 0.125f, MG)) - MB);
    const uint32_t a01 = bits(__fadd_rn(a[0], MG)) * 256u + (bits(__fadd_rn(a[1], MG)) - MB * 257u);
    const int a23 = (int)(bits(__fadd_rn(a[2], MG)) * 256u + (bits(__fadd_rn(a[3], MG)) - MB * 257u));
    const int a45 = (int)(bits(__fadd_rn(a[4], MG)) * 64u + (bits(h) - MB * 65u));    // unit 2^7
    long long V = (long long)a23 * (1 << 21) + ((long long)a45 * 128 + low);
    V += (long long)((uint64_t)(a01 << 5) << 32);
    return round_fixed(V, E, eb_out);
}

__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    // K-major operand, 128-byte swizzle, 8-row groups 1024 bytes apart
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
}

// Four consecutive-k entries into an operand's digit planes: plane s takes its
// four FP16 digits as 8 bytes at base + s * plane.
__device__ __forceinline__ void split_to(const double (&x)[4], int E, unsigned char* base, uint32_t plane)
{
    uint32_t d[DG_S][2];
    split4(x, E, d);
#pragma unroll
    for (int s = 0; s < DG_S; ++s) *reinterpret_cast<uint2*>(base + s * plane) = make_uint2(d[s][0], d[s][1]);
}

// The rare results (round_fixed asked for another look): this lane's row times
// column `col` of the CTA's range, as they stand, on the FP64 pipe.  Everything
// is taken from the arguments again, so that the main path keeps nothing for it.
template <bool BT>
__device__ __noinline__ double plain_sum(const DgArgs& a, int col)
{
    const GemmArgs<double>& g = a.g;
    const int warp = threadIdx.x >> 5;
    const int r = blockIdx.y * DG_BM + (warp & 3) * 32 + (threadIdx.x & 31);
    const int c = blockIdx.x * a.per * DG_BN + (warp >> 2) * 8 + col;
    if (r >= g.M || c >= g.N) return 0.0;
    const double* x = g.A + blockIdx.z * g.sA + r * g.lda;
    const double* y = g.B + blockIdx.z * g.sB + (BT ? c * g.ldb : c);
    const long long step = BT ? 1 : g.ldb;
    double s = 0.0;
    for (int k = 0; k < g.K; ++k) s = fma(x[k], y[k * step], s);
    return s;
}

// The same for the entries of the warp's 32 x 8 block that are set in `fix` (a
// bit per column), a row a lane.
template <bool BT>
__device__ __noinline__ void plain_block(const DgArgs& a, int col, double* st, uint32_t fix)
{
    const GemmArgs<double>& g = a.g;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = blockIdx.x * a.per * DG_BN + (warp >> 2) * 8 + col;
    const double* x = g.A + blockIdx.z * g.sA + (long long)min((int)blockIdx.y * DG_BM + (warp & 3) * 32 + lane, g.M - 1) * g.lda;
    const double* B = g.B + blockIdx.z * g.sB + (BT ? c0 * g.ldb : c0);
    const long long cs = BT ? g.ldb : 1, ks = BT ? 1 : g.ldb;
    double s[8] = {};
#pragma unroll 2
    for (int k = 0; k < g.K; ++k) {
        const double xk = x[k];
        const double* y = B + k * ks;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c0 + c < g.N) s[c] = fma(xk, y[c * cs], s[c]);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (fix >> c & 1u) st[lane * 8 + (c ^ ((lane >> 1) & 7))] = s[c];
}

// Entries of the warp's joined block that its fixed point is too coarse for
// (`fix`: a bit per column of this lane's row), summed as they stand into the
// staged block: a few by the whole warp, one after the other, more of them a row
// a lane.
template <bool BT>
__device__ __noinline__ void plain_entries(const DgArgs& a, int col, uint32_t fix, double* st)
{
    const GemmArgs<double>& g = a.g;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (__reduce_add_sync(0xffffffffu, __popc(fix)) > 8) {
        plain_block<BT>(a, col, st, fix);
        return;
    }
    const int r0 = blockIdx.y * DG_BM + (warp & 3) * 32;
    const int c0 = blockIdx.x * a.per * DG_BN + (warp >> 2) * 8 + col;
    const double* A = g.A + blockIdx.z * g.sA;
    const double* B = g.B + blockIdx.z * g.sB + (BT ? c0 * g.ldb : c0);
    const long long cs = BT ? g.ldb : 1, ks = BT ? 1 : g.ldb;
    for (int c = 0; c < 8; ++c)
        for (uint32_t m = __ballot_sync(0xffffffffu, fix >> c & 1u); m; m &= m - 1) {
            const int r = __ffs((int)m) - 1;   // inside M and N: its row and column are not zero
            const double* x = A + (long long)(r0 + r) * g.lda;
            const double* y = B + c * cs;
            double s = 0.0;
            for (int k = lane; k < g.K; k += 32) s = fma(x[k], y[k * ks], s);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) st[r * 8 + (c ^ ((r >> 1) & 7))] = s;
        }
}

// The CTA's tiles as plain FP64 sums: columns across the lanes, eight rows a warp.
// Bound by the FP64 pipe's two multiply-adds a clock (eight of a warp per load of
// B).
__device__ __noinline__ void plain_tiles(const DgArgs& a)
{
    const GemmArgs<double>& g = a.g;
    const int box = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r0 = blockIdx.y * DG_BM + warp * (DG_BM / DG_WARPS);
    const double* A = g.A + box * g.sA;
    const double* B = g.B + box * g.sB;
    double* O = g.O + box * g.sO;
    if (r0 >= g.M) return;
    for (int t = blockIdx.x * a.per; t < min((int)(blockIdx.x + 1) * a.per, a.tiles_n); ++t) {
        const int c = t * DG_BN + lane;
        if (c >= g.N) continue;
        double s[DG_BM / DG_WARPS] = {};
#pragma unroll 4
        for (int k = 0; k < g.K; ++k) {
            const double y = B[k * g.ldb + c];
#pragma unroll
            for (int u = 0; u < DG_BM / DG_WARPS; ++u)
                s[u] = fma(A[(long long)min(r0 + u, g.M - 1) * g.lda + k], y, s[u]);
        }
#pragma unroll
        for (int u = 0; u < DG_BM / DG_WARPS; ++u) {
            const int r = r0 + u;
            if (r >= g.M) break;
            double* o = O + (long long)r * g.ldo + c;
            double src = 0.0;
            if (g.mode == GM_ACC || (g.mode == GM_BWD && r < g.split)) src = *o;
            else if (g.mode == GM_FWD && r >= g.split) {
                const int pr = g.perm[box * g.sP + r];
                src = pr >= g.split ? *o : g.W[box * g.sW + (long long)pr * g.ldw + c];
            }
            *o = fma(g.alpha, s[u], src);
        }
    }
}

// BT: B is given transposed, [n][k] with k contiguous.  CHECK: the fixed point
// knows nothing below about 2^-58 of a row's times a column's scale (2^-51 at
// worst, at K = 64), so an entry is taken from it only where its sum of |a||b| is
// known to be large against that: where a factor within 2^-reach of its scale
// meets another one (a bit per factor, joined by AND), or where nothing but zeros
// meet.  Every other entry, and those of rows and columns with subnormals, are
// summed as they stand on the FP64 pipe.  LU products go by their matrix instead
// (is_wide, hps_panel.cu).
template <bool BT, bool CHECK>
__global__ void __launch_bounds__(DG_THREADS, 1)
k_digit_gemm(const __grid_constant__ DgArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t tfull[2];   // a tile's accumulators are complete
    __shared__ uint32_t tmem_sh;
    __shared__ int rowE[DG_BM];
    __shared__ int rowsrc[DG_BM];   // source of the row: -1 zero, -2 no such row, -3 the row itself, else a row of W
    __shared__ int colE[4][DG_BN];  // largest exponents of a tile's columns
    __shared__ __align__(16) int colX[2][DG_BN];  // and those less 1016, for the join
    const GemmArgs<double>& g = a.g;
    const int box = blockIdx.z;
    if (g.skip && g.skip[box]) return;
    const int t0 = blockIdx.x * a.per, cnt = min(a.per, a.tiles_n - t0);
    if (cnt <= 0) return;
    int hard = 0;   // read here, needed once the operands' loads are on their way
    if constexpr (!CHECK) hard = g.wide[box];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.y * DG_BM;
    const uint32_t sb = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* sp = smem_raw + (sb - smem_u32(smem_raw));
    const double* A = g.A + box * g.sA;
    const double* B = g.B + box * g.sB;
    double* O = g.O + box * g.sO;
    const double* W = g.W ? g.W + box * g.sW : nullptr;

    if (tid == 0) {
        mbar_init(smem_u32(&tfull[0]), 1);
        mbar_init(smem_u32(&tfull[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 4 * DG_BN) (&colE[0][0])[tid] = E_MIN;
    if (tid < DG_BM) {
        const int r = m0 + tid;
        int s = -2;
        if (r < g.M) {
            if (g.mode == GM_SET) s = -1;
            else if (g.mode == GM_ACC) s = -3;
            else if (g.mode == GM_SRC) s = r;
            else if (g.mode == GM_BWD) s = r < g.split ? -3 : -1;
            else if (r < g.split) s = -1;
            else {
                const int pr = g.perm[box * g.sP + r];
                s = pr >= g.split ? -3 : pr;
            }
        }
        rowsrc[tid] = s;
    }

    auto expo = [](double v) { return CHECK ? exp_all(v) : exp_of(v); };
    // the block of B of one tile: column lane, k = 4 warp .. +3
    double bx[4];
    const double* Bp = BT ? B + 4 * warp + (long long)lane * g.ldb : B + (long long)(4 * warp) * g.ldb + lane;
    auto load_b = [&](int tile) {
        const double* p = Bp + (BT ? (long long)tile * DG_BN * g.ldb : (long long)tile * DG_BN);
        const long long step = BT ? 1 : g.ldb;
        if ((tile + 1) * DG_BN <= g.N && g.K >= DG_K) {
#pragma unroll
            for (int u = 0; u < 4; ++u, p += step) bx[u] = *p;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u, p += step) bx[u] = tile * DG_BN + lane < g.N && 4 * warp + u < g.K ? *p : 0.0;
        }
    };
    // the strip of A: 16 threads per row, four consecutive k each
    {
        const int kg = tid & 15, k = 4 * kg;
        double x[4][4];
#pragma unroll
        for (int ps = 0; ps < 4; ++ps) {
            const int r = m0 + ps * 32 + (tid >> 4);
#pragma unroll
            for (int u = 0; u < 4; ++u) x[ps][u] = (r < g.M && k + u < g.K) ? A[(long long)r * g.lda + k + u] : 0.0;
        }
        load_b(t0);
        if constexpr (!CHECK)
            if (hard) {   // the whole box
                plain_tiles(a);
                return;
            }
        if (warp == 0) tmem_alloc(smem_u32(&tmem_sh), 512);
#pragma unroll
        for (int ps = 0; ps < 4; ++ps) {
            const int rl = ps * 32 + (tid >> 4);
            int e = E_MIN;
#pragma unroll
            for (int u = 0; u < 4; ++u) e = max(e, expo(x[ps][u]));
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
            if (kg == 0) rowE[rl] = e == E_BAD ? E_NAN : e;
            if constexpr (CHECK) sp[OFF_ST + rl * 16 + kg] = reach4(x[ps], e, a.reach);   // on its way to the row's lanes
            split_to(x[ps], e, sp + rl * 128 + (((kg >> 1) ^ (rl & 7)) << 4) + ((kg & 1) << 3), A_PLANE);
        }
    }
    __syncthreads();
    const uint32_t tmem = tmem_sh;
    const int kch = max(1, (min(g.K, DG_K) + 15) / 16);
    auto wait = [](uint64_t* bar, int use) {   // bounded: false when it gave up
        const uint32_t b = smem_u32(bar);
        if (mbar_try_wait(b, use & 1)) return true;
        const uint64_t w0 = global_ns();
        while (!mbar_try_wait(b, use & 1))
            if (global_ns() - w0 > DG_WAIT_NS) return false;
        return true;
    };
    // where this lane's eight rows of a joined block take their source: the row itself, a row of W, or nothing
    uint32_t own = 0, other = 0, valid = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int s = rowsrc[(warp & 3) * 32 + 4 * u + (lane >> 3)];
        own |= (uint32_t)(s == -3) << u;
        other |= (uint32_t)(s >= 0) << u;
        valid |= (uint32_t)(s != -2) << u;
    }
    int lost = -1;   // the tile whose wait gave up
    uint32_t near[4] = {}, flags = 0;   // CHECK: the bits of row `lane` of the warp's quarter, in the order of the columns'
    if constexpr (CHECK) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            near[i] = *reinterpret_cast<const uint32_t*>(sp + OFF_ST + ((warp & 3) * 32 + lane) * 16 + 4 * (i ^ (warp >> 2)));
    }

    // This lane's entries of a joined 32 x 8 block: rows 4 u + lane / 8, one
    // column.  A row that is its own source is added to in the L2 (one FP64 add
    // per entry, rounded as an add here would be, and nothing to wait for);
    // with the source read, added on the FP64 pipe and written back the same
    // product took 1.5 times as long.
    const int rq = (warp & 3) * 32, cg = (warp >> 2) * 8;
    double* const Or = O + (long long)(m0 + rq + (lane >> 3)) * g.ldo + cg + (lane & 7);
    const long long ostep = 4 * g.ldo;
    const bool plain = __all_sync(0xffffffffu, own == 0xffu);
    const bool unit = g.alpha == 1.0 || g.alpha == -1.0;
    const uint32_t flip = g.alpha == -1.0 ? 0x80000000u : 0u;
    double* const st = reinterpret_cast<double*>(sp + OFF_ST + warp * STAGE);

    for (int i = 0; i <= cnt; ++i) {
        if (i < cnt) {
            int e = max(max(expo(bx[0]), expo(bx[1])), max(expo(bx[2]), expo(bx[3])));
            atomicMax(&colE[i & 3][lane], e);
            __syncthreads();
            e = colE[i & 3][lane];
            split_to(bx, e, sp + OFF_B + (i & 1) * B_BUF + lane * 128 + (((warp >> 1) ^ (lane & 7)) << 4) + ((warp & 1) << 3),
                     B_PLANE);
            if constexpr (CHECK) {   // into the staging buffer of each warp that joins these columns: 16 bytes a column, words swizzled
                const unsigned char m = reach4(bx, e, a.reach);
                const int cgi = lane >> 3;
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    sp[OFF_ST + (4 * cgi + r) * STAGE + (lane & 7) * 16 + (warp ^ (cgi << 2))] = m;
            }
            if (warp == 0) {
                colE[(i + 2) & 3][lane] = E_MIN;
                colX[i & 1][lane] = e == E_BAD ? E_NAN : e - 1016;
            }
            if (i + 1 < cnt) load_b(t0 + i + 1);
            fence_proxy_async_smem();
            tc_fence_before();
            __syncthreads();
            if (tid == 0 && lost < 0) {
                tc_fence_after();
                const uint32_t d0 = tmem + (uint32_t)((i & 1) * 256);
                const uint64_t ad = sw128_desc(sb), bd = sw128_desc(sb + OFF_B + (uint32_t)(i & 1) * B_BUF);
#pragma unroll
                for (int s = 0; s < DG_S; ++s)
                    for (int kk = 0; kk < kch; ++kk)
                        mma_bf16(d0 + s * DG_BN, ad + (uint64_t)(s * (A_PLANE >> 4) + kk * 2), bd + (uint64_t)(kk * 2),
                                 f16_idesc(DG_BM, DG_BN * (DG_S - s)), (kk | s) != 0);
                mma_commit(smem_u32(&tfull[i & 1]));
            }
            __syncwarp();
        }
        // the tile's entries whose sums may be small against their scales: a bit per column of this lane's row
        const uint32_t fix = flags;
        flags = 0;
        if (CHECK && i < cnt) {
            const uint4* m = reinterpret_cast<const uint4*>(sp + OFF_ST + warp * STAGE);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint4 w = m[c];
                const uint32_t both = (near[0] & w.x) | (near[1] & w.y) | (near[2] & w.z) | (near[3] & w.w);
                flags |= (uint32_t)(both != 0 && (both & 0x0F0F0F0Fu) == 0) << c;
            }
            __syncwarp();
        }
        if (i == 0) continue;
        // join tile i - 1: the warp's quarter of the rows, eight of the 32
        // columns, four at a time
        const int j = i - 1, buf = j & 1;
        const int col = (t0 + j) * DG_BN + cg + (lane & 7);
        const bool in = col < g.N;
        double src[8];
        if (g.mode == GM_SRC) {   // consecutive rows of W
            const double* w = W + (long long)(m0 + rq + (lane >> 3)) * g.ldw + col;
#pragma unroll
            for (int u = 0; u < 8; ++u) src[u] = in && (other >> u & 1) ? w[4 * u * g.ldw] : 0.0;
        }
        if (lost < 0 && !wait(&tfull[buf], j >> 1)) lost = j;
        tc_fence_after();
        const int Ea = lost < 0 ? rowE[rq + lane] : E_NAN;
#pragma unroll
        for (int h = 0; h < 8; h += 4) {
            uint32_t v[DG_S][4];
#pragma unroll
            for (int t = 0; t < DG_S; ++t)
                tmem_ld4(tmem + ((uint32_t)rq << 16) + (uint32_t)(buf * 256 + t * DG_BN + cg + h), v[t]);
            const int4 ex = *reinterpret_cast<const int4*>(&colX[buf][cg + h]);
            const int E[4] = {Ea + ex.x, Ea + ex.y, Ea + ex.z, Ea + ex.w};
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            int eb[4];
            bool odd = false;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float q[DG_S];
#pragma unroll
                for (int t = 0; t < DG_S; ++t) q[t] = __uint_as_float(v[t][c]);
                st[lane * 8 + ((h + c) ^ ((lane >> 1) & 7))] = join(q, E[c], eb[c]);
                odd |= (unsigned)eb[c] > 2045u;
            }
            if (odd) {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if ((unsigned)eb[c] > 2045u)
                        st[lane * 8 + ((h + c) ^ ((lane >> 1) & 7))] = plain_sum<BT>(a, j * DG_BN + h + c);
            }
        }
        __syncwarp();
        if (CHECK && __any_sync(0xffffffffu, fix != 0)) {
            plain_entries<BT>(a, j * DG_BN, fix, st);
            __syncwarp();
        }
        {
            double* p = Or + (long long)(t0 + j) * DG_BN;
            auto joined = [&](int u) {
                const int rl = 4 * u + (lane >> 3);
                return st[rl * 8 + ((lane & 7) ^ ((rl >> 1) & 7))];
            };
            auto scaled = [&](double r) {
                return unit ? __hiloint2double((int)((uint32_t)__double2hiint(r) ^ flip), __double2loint(r)) : g.alpha * r;
            };
            if (g.mode == GM_SRC) {
#pragma unroll
                for (int u = 0; u < 8; ++u, p += ostep)
                    if (in && (valid >> u & 1)) *p = fma(g.alpha, joined(u), src[u]);
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u, p += ostep) {
                    double r = scaled(joined(u));
                    if (plain || (own >> u & 1)) {
                        if (in) atomicAdd(p, r);
                    } else if (in && (valid >> u & 1)) {
                        if (other >> u & 1) r += W[(long long)rowsrc[rq + 4 * u + (lane >> 3)] * g.ldw + col];
                        *p = r;
                    }
                }
            }
        }
        __syncwarp();
        tc_fence_before();
    }
    if (lost >= 0) {
        if (lane == 0 && g.status) g.status[box] = HPS_ETIMEOUT;
        // no tile is issued any more; the one that was lost and the next, already issued, end before TMEM is freed
        if (warp == 0)
            for (int t = lost; t < min(lost + 2, cnt); ++t) wait(&tfull[t & 1], t >> 1);
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

}  // namespace

void launch_digit_gemm(const GemmArgs<double>& in, bool b_transposed, int nbox, cudaStream_t st)
{
    GemmArgs<double> g = in;
    if (g.M <= 0 || g.N <= 0 || nbox <= 0) return;
    auto kern = b_transposed ? k_digit_gemm<true, true> : g.wide ? k_digit_gemm<false, false> : k_digit_gemm<false, true>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DG_SMEM);
    DgArgs a;
    // A product by itself (B transposed: factors given by the caller) is held to
    // the K 2^-53 sum |a||b| of an FP64 sum: the fixed point is off by at most
    // K 2^-57 of the scales' product, which is that where the sum is 2^-4 of it.
    // Products with interface factors keep 29 bits of every entry (36 typically).
    a.reach = b_transposed ? 2 : 11;
    a.tiles_n = (g.N + DG_BN - 1) / DG_BN;
    const int tiles_m = (g.M + DG_BM - 1) / DG_BM;
    // Columns of a strip are shared out so that the CTAs fill the SMs evenly: a
    // CTA costs about three tiles (its strip of A, the pipeline's ends) plus
    // its own, and the makespan is the waves times that.
    const long long strips = (long long)tiles_m * nbox;
    const int sms = sm_count();
    long long best = -1;
    int ns_best = 1;
    for (int ns = 1; ns <= std::min(a.tiles_n, 32); ++ns) {
        const long long waves = (strips * ns + sms - 1) / sms, cost = waves * (3 + (a.tiles_n + ns - 1) / ns);
        if (best < 0 || cost < best) { best = cost; ns_best = ns; }
    }
    a.per = (a.tiles_n + ns_best - 1) / ns_best;
    dim3 grd((unsigned)((a.tiles_n + a.per - 1) / a.per), (unsigned)tiles_m, (unsigned)nbox);
    // K beyond one product's 64: further passes add to what the first wrote.
    for (int k0 = 0; k0 < g.K || k0 == 0; k0 += DG_K) {
        a.g = g;
        a.g.K = std::max(0, std::min(DG_K, g.K - k0));
        a.g.A = g.A + k0;
        a.g.B = b_transposed ? g.B + k0 : g.B + (long long)k0 * g.ldb;
        if (k0 && in.mode == GM_SRC) {   // read and written back (O may be mapped host memory), not added to in the L2
            a.g.W = in.O; a.g.ldw = in.ldo; a.g.sW = in.sO;
        } else if (k0) {
            a.g.mode = GM_ACC;
        }
        prof_begin(KC_UPDATE_TC, st);
        kern<<<grd, DG_THREADS, DG_SMEM, st>>>(a);
        prof_end(KC_UPDATE_TC, st, 2.0 * nbox * g.M * (double)g.N * a.g.K,
                 (double)nbox * ((double)g.M * a.g.K + (double)a.g.K * g.N + 2.0 * g.M * g.N) * 8);
    }
}

}  // namespace hps
