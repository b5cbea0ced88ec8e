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
// So the only roundings are those three; a plain FP64 sum rounds K times.
// Against a higher-precision solve, the LU built on these products is as close
// as or closer than the one on FP64 multiply-adds (tests/test_gpu_digit.py).
// A row or column that holds an infinity or a NaN gives NaN throughout.
//
// Bound and layout.  One CTA of 512 threads per SM takes a 128-row strip of A
// (split once, 128 KiB of digits in shared memory) across a range of column
// tiles of 32.  Per tile all threads split the 64 x 32 block of B (double
// buffered), one thread issues 32 MMAs (A digit i against the stacked digits
// 0..7-i of B, N = 32 (8 - i): the diagonals t land in consecutive TMEM
// columns), and while they run every warp joins 32 x 8 outputs of the tile
// before (TMEM holds two tiles of 8 x 32 columns, all 512).  A tile's 4096
// outputs need 2176 tensor-core clocks, about 2500 clocks of issue and
// 2048 clocks of FP64 adds, and move 64 KB of O: the three are balanced, with
// HBM close behind at K = 64.  Measured against the CUDA-core FP64 product:
// 512 boxes at p = 12 (DtN, particular and reconstruction) 1001 -> 147 ms for
// the whole call, cross-term leaves 225 -> 59 ms.
#include <algorithm>

#include "hps_internal.h"
#include "hps_ptx.cuh"

#include <cuda_fp16.h>

namespace hps {

namespace {

constexpr int DG_S = 8;                                // digits of an operand
constexpr int DG_BM = 128, DG_BN = 32, DG_K = 64;      // tile
constexpr int DG_THREADS = 512, DG_WARPS = DG_THREADS / 32;
constexpr uint32_t A_PLANE = DG_BM * 128;              // one digit of A: rows of 64 FP16 (128 B, 128B swizzle)
constexpr uint32_t B_PLANE = DG_BN * 128;
constexpr uint32_t B_BUF = DG_S * B_PLANE;
constexpr uint32_t STAGE = 32 * 8 * 8;                 // per warp: 32 x 8 results
constexpr uint32_t OFF_B = DG_S * A_PLANE, OFF_ST = OFF_B + 2 * B_BUF;
constexpr size_t DG_SMEM = OFF_ST + DG_WARPS * STAGE + 1024;
constexpr uint64_t DG_WAIT_NS = 2000000000ull;
constexpr int E_MIN = 1;     // scale exponent of a row or column of zeros (subnormal entries count as zero)
constexpr int E_BAD = 2047;  // an infinity or NaN in the row or column: its scale is then kept as E_NAN
constexpr int E_NAN = 1 << 20;

struct DgArgs {
    GemmArgs<double> g;
    int tiles_n, per;   // column tiles, and how many of them a CTA takes
};

__device__ __forceinline__ int exp_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Four consecutive-k entries under the scale exponent E: digit plane s gets the
// four FP16 digits as 8 bytes at base + s * plane.
__device__ __forceinline__ void split4(const double (&x)[4], int E, unsigned char* base, uint32_t plane)
{
    uint32_t w[4][2];
    __half2 sg[2], off[2], off0[2];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint32_t hi = (uint32_t)__double2hiint(x[u]), lo = (uint32_t)__double2loint(x[u]);
        const int e = (int)((hi >> 20) & 0x7ffu);
        const int d = e ? min(E - e, 63) : 63;   // zero (and subnormal) entries: all digits zero
        const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
        const uint64_t m = ((((uint64_t)mh << 32) | lo) << 9) >> d;
        const uint64_t b = m + 0x0080808080808080ull;   // balanced digits: byte - 128 below the leading one
        w[u][0] = (uint32_t)b;
        w[u][1] = (uint32_t)(b >> 32);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // +-1 of the two entries, and the biases of 1024 + byte that belong to them
        const uint32_t h0 = (uint32_t)__double2hiint(x[2 * h]), h1 = (uint32_t)__double2hiint(x[2 * h + 1]);
        const uint32_t sb = ((h0 >> 16) & 0x8000u) | (h1 & 0x80000000u);
        const uint32_t one = 0x3C003C00u ^ sb, o1152 = 0xE480E480u ^ sb, o1024 = 0xE400E400u ^ sb;
        sg[h] = *reinterpret_cast<const __half2*>(&one);
        off[h] = *reinterpret_cast<const __half2*>(&o1152);
        off0[h] = *reinterpret_cast<const __half2*>(&o1024);
    }
#pragma unroll
    for (int s = 0; s < DG_S; ++s) {
        const int byte = 7 - s;   // plane 0 holds the leading digit
        uint32_t r[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t a = w[2 * h][byte >> 2], b = w[2 * h + 1][byte >> 2];
            uint32_t v = __byte_perm(a, b, (uint32_t)(byte & 3) | ((uint32_t)(4 + (byte & 3)) << 8));
            v = (v & 0x00FF00FFu) | 0x64006400u;   // FP16 1024 + byte
            const __half2 d = __hfma2(*reinterpret_cast<const __half2*>(&v), sg[h], s == 0 ? off0[h] : off[h]);
            r[h] = *reinterpret_cast<const uint32_t*>(&d);
        }
        *reinterpret_cast<uint2*>(base + s * plane) = make_uint2(r[0], r[1]);
    }
}

// Sum of acc_t 2^(45 - 8 t) (unit 2^-57 of the scales' product 2^(E - 1016 ..))
// rounded once to FP64.  The accumulators are turned to integers by adding
// 1.5 2^23 (the conversion instruction runs at 16 lanes a clock and took 93 %
// of the kernel's time): exact below 2^22, which holds for t <= 4 (the leading
// digits are at most 64).  t = 5 is first cut to a multiple of 4, whose rest
// joins t = 6, 7; those only need to be right to a fraction of the unit, so
// their sum is taken in FP32 (an error below 2^-4 units).
// E: biased exponents of the two scales, less 1016.  A result outside the
// normal range (or of a row or column with an infinity or NaN) sets `odd`, and
// finish_odd gives it; the common path has no branch, so that the eight joins
// of a thread overlap.
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
    const int sm = (int)(V >> 63);
    uint64_t u = (uint64_t)((V ^ (long long)sm) - (long long)sm);
    const int lz = __clzll((long long)u);              // 1 .. 63, 64 for zero
    u <<= (lz - 1) & 63;
    u += 512;                                          // the leading bit is bit 62: 53 bits stay
    int eb = E - lz;
    uint64_t r = (u >> 10) + ((uint64_t)(uint32_t)eb << 52);
    r |= (uint64_t)((uint32_t)sm & 0x80000000u) << 32;
    const bool zero = lz == 64 && E < (1 << 19);
    eb_out = zero ? 0 : lz == 64 ? 4096 : eb;
    return __longlong_as_double(zero ? 0ll : (long long)r);
}

// The rare results: `r` has the sign, E and eb are those of its join.
__device__ __noinline__ double finish_odd(double r, int E, int eb)
{
    if ((unsigned)eb <= 2045u) return r;
    if (E >= (1 << 19)) return __longlong_as_double(0x7FF8000000000000ll);   // an infinity or NaN went in
    const long long sg = __double_as_longlong(r) & (long long)0x8000000000000000ull;
    return __longlong_as_double(sg | (eb < 0 ? 0ll : 0x7FF0000000000000ll));
}

__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    // K-major operand, 128-byte swizzle, 8-row groups 1024 bytes apart
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr));
}

// BT: B is given transposed, [n][k] with k contiguous.
template <bool BT>
__global__ void __launch_bounds__(DG_THREADS, 1)
k_digit_gemm(const DgArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t tfull[2];
    __shared__ uint32_t tmem_sh;
    __shared__ int rowE[DG_BM];
    __shared__ int rowsrc[DG_BM];   // source of the row: -1 zero, -2 no such row, -3 the row itself, else a row of W
    __shared__ int colE[4][DG_BN];  // largest exponents of a tile's columns
    __shared__ int colX[2][DG_BN];  // the same, less 1016, for the join
    const GemmArgs<double>& g = a.g;
    const int box = blockIdx.z;
    if (g.skip && g.skip[box]) return;
    const int t0 = blockIdx.x * a.per, cnt = min(a.per, a.tiles_n - t0);
    if (cnt <= 0) return;
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
    if (warp == 0) tmem_alloc(smem_u32(&tmem_sh), 512);
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

    // the block of B of one tile: column n0 + lane, k = 4 warp .. +3
    double bx[4];
    auto load_b = [&](int tile) {
        const int n = tile * DG_BN + lane, k = 4 * warp;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            bx[u] = 0.0;
            if (n < g.N && k + u < g.K) bx[u] = BT ? B[(long long)n * g.ldb + k + u] : B[(long long)(k + u) * g.ldb + n];
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
#pragma unroll
        for (int ps = 0; ps < 4; ++ps) {
            const int rl = ps * 32 + (tid >> 4);
            int e = E_MIN;
#pragma unroll
            for (int u = 0; u < 4; ++u) e = max(e, exp_of(x[ps][u]));
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
            if (kg == 0) rowE[rl] = e == E_BAD ? E_NAN : e;
            split4(x[ps], e, sp + rl * 128 + (((kg >> 1) ^ (rl & 7)) << 4) + ((kg & 1) << 3), A_PLANE);
        }
    }
    __syncthreads();
    const uint32_t tmem = tmem_sh;
    // where this lane's eight rows of a joined block take their source: the row itself, a row of W, or nothing
    uint32_t own = 0, other = 0, valid = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int s = rowsrc[(warp & 3) * 32 + 4 * u + (lane >> 3)];
        own |= (uint32_t)(s == -3) << u;
        other |= (uint32_t)(s >= 0) << u;
        valid |= (uint32_t)(s != -2) << u;
    }
    const int kch = max(1, (min(g.K, DG_K) + 15) / 16);
    bool ok = true;

    for (int i = 0; i <= cnt; ++i) {
        if (i < cnt) {
            int e = max(max(exp_of(bx[0]), exp_of(bx[1])), max(exp_of(bx[2]), exp_of(bx[3])));
            atomicMax(&colE[i & 3][lane], e);
            __syncthreads();
            e = colE[i & 3][lane];
            split4(bx, e, sp + OFF_B + (i & 1) * B_BUF + lane * 128 + (((warp >> 1) ^ (lane & 7)) << 4) + ((warp & 1) << 3),
                   B_PLANE);
            if (warp == 0) {
                colE[(i + 2) & 3][lane] = E_MIN;
                colX[i & 1][lane] = e == E_BAD ? E_NAN : e - 1016;
            }
            if (i + 1 < cnt) load_b(t0 + i + 1);
            fence_proxy_async_smem();
            tc_fence_before();
            __syncthreads();
            if (tid == 0) {
                tc_fence_after();
                const uint32_t d0 = tmem + (uint32_t)((i & 1) * 256);
                const uint32_t bb = sb + OFF_B + (uint32_t)(i & 1) * B_BUF;
                for (int kk = 0; kk < kch; ++kk) {
                    const uint64_t bd = sw128_desc(bb + kk * 32);
#pragma unroll
                    for (int s = 0; s < DG_S; ++s)
                        mma_bf16(d0 + s * DG_BN, sw128_desc(sb + s * A_PLANE + kk * 32), bd,
                                 f16_idesc(DG_BM, DG_BN * (DG_S - s)), (kk | s) != 0);
                }
                mma_commit(smem_u32(&tfull[i & 1]));
            }
        }
        if (i == 0) continue;
        // join tile i - 1: warp's lane quarter rows, eight of the 32 columns
        const int j = i - 1, buf = j & 1, rq = (warp & 3) * 32, cg = (warp >> 2) * 8;
        const int n0 = (t0 + j) * DG_BN + cg;
        const int col = n0 + (lane & 7);
        double src[8];
        const bool in = col < g.N;
        double* Oc = O + (long long)(m0 + rq + (lane >> 3)) * g.ldo + col;
        const long long ostep = 4 * g.ldo;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            src[u] = 0.0;
            if (in && (own >> u & 1)) src[u] = Oc[u * ostep];
        }
        if (other && in) {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (other >> u & 1) src[u] = W[(long long)rowsrc[rq + 4 * u + (lane >> 3)] * g.ldw + col];
        }
        if (ok && !mbar_try_wait(smem_u32(&tfull[buf]), (j >> 1) & 1)) {
            const uint64_t w0 = global_ns();
            while (!mbar_try_wait(smem_u32(&tfull[buf]), (j >> 1) & 1))
                if (global_ns() - w0 > DG_WAIT_NS) { ok = false; break; }
        }
        tc_fence_after();
        uint32_t v[DG_S][8];
#pragma unroll
        for (int t = 0; t < DG_S; ++t)
            tmem_ld8(tmem + ((uint32_t)rq << 16) + (uint32_t)(buf * 256 + t * DG_BN + cg), v[t]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        const int Ea = ok ? rowE[rq + lane] : E_NAN;
        double* st = reinterpret_cast<double*>(sp + OFF_ST + warp * STAGE);
        int eb[8];
        bool odd = false;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            float q[DG_S];
#pragma unroll
            for (int t = 0; t < DG_S; ++t) q[t] = __uint_as_float(v[t][c]);
            st[lane * 8 + (c ^ ((lane >> 1) & 7))] = join(q, Ea + colX[buf][cg + c], eb[c]);
            odd |= (unsigned)eb[c] > 2045u;
        }
        if (odd) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                double& r = st[lane * 8 + (c ^ ((lane >> 1) & 7))];
                r = finish_odd(r, Ea + colX[buf][cg + c], eb[c]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int rl = 4 * u + (lane >> 3);
            const double r = fma(g.alpha, st[rl * 8 + ((lane & 7) ^ ((rl >> 1) & 7))], src[u]);
            if (in && (valid >> u & 1)) Oc[u * ostep] = r;
        }
        tc_fence_before();
    }
    if (!ok && lane == 0 && g.status) g.status[box] = HPS_ETIMEOUT;
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

int sm_count()
{
    static int n = 0;   // the library serves one kind of GPU; 152 on GB300
    if (!n) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            n = 152;
    }
    return n;
}

}  // namespace

void launch_digit_gemm(const GemmArgs<double>& in, bool b_transposed, int nbox, cudaStream_t st)
{
    GemmArgs<double> g = in;
    if (g.M <= 0 || g.N <= 0 || nbox <= 0) return;
    auto kern = b_transposed ? k_digit_gemm<true> : k_digit_gemm<false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DG_SMEM);
    DgArgs a;
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
        if (k0) a.g.mode = GM_ACC;
        prof_begin(KC_UPDATE_TC, st);
        kern<<<grd, DG_THREADS, DG_SMEM, st>>>(a);
        prof_end(KC_UPDATE_TC, st, 2.0 * nbox * g.M * (double)g.N * a.g.K,
                 (double)nbox * ((double)g.M * a.g.K + (double)a.g.K * g.N + 2.0 * g.M * g.N) * 8);
    }
}

}  // namespace hps
