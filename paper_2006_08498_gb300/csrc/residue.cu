// FP64-accurate complex products on the tensor cores in residue arithmetic
// (the Chinese remainder form of the Ozaki scheme: Ozaki, Uchino, Imamura,
// "Ozaki scheme II", 2025).  It is the Chebyshev filter's product H Y (Sec. 3
// and the Supplement's "Filter" item: a repeated HEMM) and the Lanczos and
// Rayleigh-Ritz products with H of the FP64 mode on full storage.
//
// Representation.  Row i of A is scaled by a power of two so that its 2-norm
// is at most 2^kAlpha, column j of B so that its is at most 2^kBeta, and both
// are rounded to integers.  By Cauchy-Schwarz the real and imaginary parts of
// every element of the integer product are below 2^(kAlpha + kBeta) < P / 2,
// P the product of kNMod pairwise coprime moduli of at most 8 bits, so they
// are determined by their residues.  For each modulus the residues, balanced
// in [-128, 127], are exact in FP16, and so are their products' FP32 sums
// over 512 terms (kRange): the tensor cores do exact arithmetic.
//
// Why residues.  With slices of 8 bits an FP64-accurate product takes every
// pair of slices of the two operands (21 pairs of 48-bit operands with the
// small ones left out); residues multiply modulus by modulus, 14 products for
// operands of 54 bits: 14 x 8 = 112 tensor flops per complex multiply-add,
// against 168.  And modulo p the complex product can take three real ones (Gauss)
// instead of four, without the cancellation that form has in floating point:
//   T0 = Ar Br, T1 = Ai Bi, T2 = (Ar + Ai)(Br + Bi);
//   Re = T0 - T1, Im = T2 - T0 - T1  (mod p), 14 x 6 = 84.
// Wide tiles, bound by the tensor cores (and their power), take three; narrow ones
// take four, with fewer operands and accumulators to hand on.
//
// Accuracy.  The only rounding is that of the operands (and one FP64 rounding of the
// result): an rms error of 2^-53.8 of the norms' product ||h_i|| ||y_j|| at most, measured 2^-54.1
// from N = 256 to 40000.  The slices, which round against a line's largest entry and
// leave partial sums out, have 2^-46.4 to 2^-46.9 on exciton matrices (one large entry a
// row) and 2^-49.7 (N = 256) to 2^-52.1 (N = 40000) on matrices of even entries.  13 moduli
// and operands of 51 and 50 bits, 4 to 7 % less time, have 2^-50.4 on both, less than the
// slices on the latter.
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>

#include "gen_element.cuh"
#include "kernels.h"
#include "residue.h"
#include "rotation.h"
#include "tc_common.cuh"

namespace {

// The kernels of a product follow one another without the gap of a launch: each
// may be set up while the one before it drains (programmatic dependent launch),
// waits for that one's end before it touches memory, and lets the next one be set up.
// (No timing events between them either, outside solves.)  With 13 moduli: N = 256, 30
// columns 55 -> 47 us a product with its preparation; filter N = 2000, 75 columns
// 2.05 -> 1.78 ms.
__device__ __forceinline__ void follow() {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}
template <class... P, class... A>
void launch_next(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // an error shows at the caller's cudaGetLastError
}

// ------------------------------------------------------------ the moduli
// The product with H takes the first kNMod; the general products (kGMod below),
// which stand in for native FP64, two more and operands of kGBits bits.
constexpr int kNMod = 14, kGMod = 15;
constexpr int kAlpha = 54, kBeta = 54, kGBits = 58;
constexpr int kMod[kGMod] = {256, 253, 251, 249, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197};

constexpr int gcd_of(int a, int b) { return b == 0 ? a : gcd_of(b, a % b); }
constexpr bool coprime() {
    for (int i = 0; i < kGMod; i++)
        for (int j = 0; j < i; j++)
            if (gcd_of(kMod[i], kMod[j]) != 1) return false;
    return true;
}
static_assert(coprime(), "pairwise coprime moduli");
constexpr unsigned __int128 modulus_product(int n) {
    unsigned __int128 P = 1;
    for (int i = 0; i < n; i++) P *= (unsigned)kMod[i];
    return P;
}
// 2^(kAlpha + kBeta) plus 20 % (norm estimates and the operands' rounding) below P / 2
static_assert(modulus_product(kNMod) / 2 > ((unsigned __int128)6 << (kAlpha + kBeta)) / 5 &&
                  modulus_product(kGMod) / 2 > ((unsigned __int128)6 << (2 * kGBits)) / 5, "range of the product");

// Constants of one modulus.  A residue of the 64-bit integer X + 2^63 (bytes
// b_0..b_7): v = sum_i b_i (256^i mod p) + k0 - 12582912 by two 4-byte dot
// products, below 2^20; started at k0 they leave the bit pattern of the float
// 1.5 2^23 + v, an integer F below 2^24 that k0 makes congruent to X.  Then r = F -
// p rint(F / p) in FP32 (two FMAs and an addition, exact; |r| <= p / 2 + 1, so at
// most 127 for p <= 253, and 256 divides exactly), and the low byte of r + 128 +
// 2^23 is the residue as it is stored: b in [0, 255] stands for b - 128.
// (The same with an integer multiply-high and multiply in place of the FP32
// steps: 278 instructions per element of A for 26 residues, 178 of them on one
// of the two FMA pipes.)
struct ModConst {
    uint32_t clo, chi, k0;
    float pf, inv;
    uint32_t w[2][3];       // W = round(2^96 ((P/p)^-1 mod p) / p), low word first: of kNMod moduli, and of all kGMod
};
struct ModTable {
    ModConst m[kGMod];
    unsigned long long bias[2][2];     // 128 sum_m W_m of either: low and high 64 bits
};
constexpr unsigned inverse_of_rest(int i, int n) {     // (P / p_i)^-1 mod p_i, P of the first n
    const unsigned p = (unsigned)kMod[i];
    unsigned q = 1;
    for (int j = 0; j < n; j++)
        if (j != i) q = q * ((unsigned)kMod[j] % p) % p;
    unsigned v = 1;
    while (q * v % p != 1) v++;
    return v;
}
constexpr ModTable make_table() {
    ModTable t{};
    unsigned __int128 bias[2] = {};
    for (int i = 0; i < kGMod; i++) {
        const unsigned p = (unsigned)kMod[i];
        unsigned c = 1 % p, cc[8] = {};
        for (int b = 0; b < 8; b++) {
            cc[b] = c;
            c = c * 256u % p;
        }
        t.m[i].clo = cc[0] | cc[1] << 8 | cc[2] << 16 | cc[3] << 24;
        t.m[i].chi = cc[4] | cc[5] << 8 | cc[6] << 16 | cc[7] << 24;
        // F = 12582912 + (k0 - 0x4B400000) + sum: congruent to X
        const unsigned two63 = cc[7] * 128u % p, base = 12582912u % p;
        t.m[i].k0 = 0x4B400000u + (2 * p - two63 - base) % p;
        t.m[i].pf = (float)p;
        t.m[i].inv = 1.0f / (float)p;
        for (int set = 0; set < 2; set++) {
            const int n = set == 0 ? kNMod : kGMod;
            if (i >= n) continue;
            const unsigned __int128 W = (((unsigned __int128)inverse_of_rest(i, n) << 96) + p / 2) / p;
            for (int k = 0; k < 3; k++) t.m[i].w[set][k] = (uint32_t)(W >> (32 * k));
            bias[set] += 128 * W;
        }
    }
    for (int set = 0; set < 2; set++)
        for (int k = 0; k < 2; k++) t.bias[set][k] = (unsigned long long)(bias[set] >> (64 * k));
    return t;
}
__constant__ ModTable kTab = make_table();

// The element is F / 2^96 P with F = sum_m W_m r_m modulo 2^96 as a signed
// number: the fraction of sum_m r_m inv_m / p_m, to 2^-84 of the range, so that an
// element far below its norms' product keeps its FP64 digits (with 64 bits the sum over
// the K splits' residues costs up to 2^-52 of the norms' product).  P as a 64-bit
// mantissa: P = mant 2^exp.
constexpr unsigned long long mantissa(int n, int e) {
    return (unsigned long long)((modulus_product(n) + ((unsigned __int128)1 << (e - 1))) >> e);
}
constexpr int kHExp = 47, kGExp = 54;
constexpr unsigned long long kHMant = mantissa(kNMod, kHExp), kGMant = mantissa(kGMod, kGExp);
static_assert(kHMant >> 63 == 1 && kGMant >> 63 == 1, "normalised");

// ------------------------------------------------------------ the tiling
constexpr int kRows = 128;         // rows of a CTA (TMEM lanes, MMA M)
constexpr int kMaxW = 144;         // complex columns of a CTA at most
constexpr int kChunk = 64;         // K elements of a stage (one swizzle row of FP16)
constexpr int kGaussW = 112;       // three real products above this width, four up to it
constexpr int kRange = 8;          // the exact range of an FP32 sum of two terms per K (T2, Re, Im), in chunks
constexpr int kMaxUnitChunks = 224;           // a drain thread's packed sums
constexpr int kAStage = 2 * kRows * kChunk;   // Re and Im residues, one byte each
constexpr int kPack = 8192;        // a drain thread keeps Re + kPack Im in one integer
constexpr int kDrainWarps = 8;
constexpr int kTmemCols = 512;
// Tensor memory holds three accumulators of a launch's widest tile (Gauss: one per
// product; four products: Re, Im, and the one that is being drained) and, in the
// rest, the ring of A operand stages, which covers the latency between an MMA's
// reading a stage and the MMA that reads its next contents.  Gauss: a stage is 16
// columns, K = 32 of one of the three operands, 5 beside 144 columns.  Four
// products: Re and Im of a chunk (64 columns) or of half of it.
constexpr int kMaxSlots = 16;
constexpr int kBars = 32;          // Gauss: barriers of the stages, as a ring (a power of two, above kMaxSlots)

// Variants by the widest column tile of a launch.  Converting A costs the same
// whatever the width, so a narrow tile is bound by the converters: it has more
// of them, which the drain threads' registers (one packed sum per column) allow.
// Warpgroups (4 warps, one per TMEM quadrant): copies and MMAs; kConv converter
// groups; two drain groups.  Registers a thread: R0, RC, RD (setmaxnreg moves
// them from the others to the drain groups) of RL at launch; 0: no move.
// H: stages of A a chunk takes (four products), 0: Gauss.  With 13 moduli, N = 8000, us at 16, 48, 80,
// 96, 112, 128, 144 columns: Gauss 295 314 351 375 443 455 481, four products 240 266
// 324 359 407 444 508 (H's residues cross HBM in 248); twenty products of 140
// columns at N = 20000, where the power limit counts too: 66.9 and 71.6 ms.
template <int W, int CONV, int SA, int SB, int HOLD, int H, int RL, int R0, int RC, int RD>
struct RsCfg {
    static constexpr int kW = W;                   // columns of a tile at most
    static constexpr bool kGauss = H == 0;
    static constexpr int kProducts = kGauss ? 3 : 2;   // accumulators, MMA warps and parts of B
    static constexpr int kConv = CONV;
    static constexpr int kThreads = 32 * (4 + 4 * CONV + kDrainWarps);
    static constexpr int kSA = SA, kSB = SB;       // stages of A's bytes and of B
    static constexpr int kBStage = kProducts * W * kChunk * 2;
    static constexpr int kSmem = SA * kAStage + SB * kBStage + 1024;
    static constexpr int kHold = HOLD;             // granules of 8 columns a drain thread loads at once
    static constexpr int kH = kGauss ? 2 : H, kCols = kGauss ? 16 : 64 / kH;   // stages of A and their columns
    static constexpr int kR0 = R0, kRC = RC, kRD = RD;
    static_assert(128 * (R0 + CONV * RC + 2 * RD) <= kThreads * RL && 65536 / kThreads >= RL, "register split");
    static_assert(kSmem <= 230500 && 2 * HOLD >= W / 16, "resources");
    static constexpr int kMinSlots = (kTmemCols - 3 * W) / kCols;
    // H = 1: with an odd number of groups a stage of A's bytes goes to different ones in
    // turn.  A group at chunk m has seen those up to m - 2 - slots used, which covers the
    // stage's last contents (chunk m - SA), so no older phase answers its wait; such
    // variants have tiles above 48 columns.
    static_assert(H != 1 || CONV % 2 == 0 || SA >= 2 + (kTmemCols - 3 * 64) / 64, "phases of A's stages");
    // a converter group's step along the rings: one turn at most
    static_assert(CONV >= 2 && (H == 1 ? (CONV + 1) / 2 : kGauss ? 3 * (CONV - 1) : CONV) <= kMinSlots && (CONV + 1) / 2 <= SA, "rings");
};
using RsGauss = RsCfg<144, 2, 3, 3, 6, 0, 96, 48, 80, 136>;
using RsWide = RsCfg<112, 2, 5, 4, 6, 2, 96, 48, 80, 136>;
using RsMid = RsCfg<96, 3, 7, 4, 6, 1, 80, 48, 64, 112>;
using RsNarrow = RsCfg<48, 4, 8, 6, 3, 1, 72, 0, 0, 0>;
static_assert((long long)kRange * kChunk * 128 * 256 <= (1ll << 24) &&
                  2ll * kRange * kChunk * 128 * 128 <= (1ll << 24), "exact FP32 sums");
static_assert((kMaxUnitChunks / (2 * kRange) + 1) * 2 * 128 < kPack / 2 &&
                  (kMaxUnitChunks / kRange + 1) * 128 < kPack / 2, "packed sums");
static_assert(kRange == 8, "drain pattern");
// Gauss: the accumulators are drained after chunk c of a unit of nc: T0 when c % 16
// is 15, T1 when it is 10, T2 (whose operand Ar + Ai is twice as large) when it is
// 5 or 13, and all three after the last chunk: spread over time, so that each
// drain is over before the next is due.
__device__ __forceinline__ bool range_end(int t, int c) {
    return t == 0 ? (c & 15) == 15 : t == 1 ? (c & 15) == 10 : (c & 7) == 5;
}
constexpr uint64_t kWindDownNs = 2000000000ull;

// Work per CTA: one modulus, 128 rows, w <= 144 columns, the K chunks of one
// split.  Persistent, one CTA per SM, units walked by modulus (slowest), split,
// row tile and column tile (fastest), so that the CTAs running at one time
// read one modulus' operand (L2) and different rows of A.
//
//   warp 0      copies A's bytes (16 KB per chunk, untiled) into a ring of stages;
//   warps 1-3   Gauss: copy a part of B each (FP16, one TMA box per chunk) and issue
//               the MMAs of its product; four products: 1 and 2 issue those of
//               Re (Ar Br, then -Ai Bi: the descriptor negates) and of Im (Ar Bi,
//               Ai Br), 3 copies B (Re and Im in one box); per chunk 4 K steps;
//   converters  turn A's bytes into FP16 pairs (a byte permute makes 1024 + b,
//               one subtraction b - 128), with Gauss add Re and Im for the third
//               product, and store them into tensor memory: one byte per residue
//               crosses HBM and shared memory, and the MMA reads only B from
//               shared memory;
//   the last 8  drain the accumulators within their range: reduce modulo p in FP32
//               (exact: two FMAs and an addition, two values an instruction)
//               and add into one packed integer per output.
template <class Cfg>
__global__ void __launch_bounds__(Cfg::kThreads, 1) k_res_zgemm(const __grid_constant__ RsBatch bt) {
    constexpr int kConvWarps = 4 * Cfg::kConv;
    constexpr bool kGauss = Cfg::kGauss;
    constexpr int kH = Cfg::kH, kCols = Cfg::kCols, kP = Cfg::kProducts;
    constexpr int kSA = Cfg::kSA, kSB = Cfg::kSB, kBStage = Cfg::kBStage, kConvGroups = Cfg::kConv;
    extern __shared__ uint8_t smraw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    uint8_t *sB = sm, *sA = sm + kSB * kBStage;
    __shared__ uint64_t fullA[kSA], emptyA[kSA], fullB[3 * kSB], emptyB[3 * kSB];   // B, Gauss: per product
    __shared__ uint64_t accFull[3], accEmpty[AccState::kEnds], mmaDone;   // empty, Gauss: per product; else per end
    __shared__ __align__(2 * kBars * 8) uint64_t aBars[2 * kBars];   // stages of A: full, then empty
    uint64_t *aFull = aBars, *aEmpty = aBars + kBars;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    const int units = bt.units;
    const uint32_t stride = (uint32_t)bt.stride, slots = (uint32_t)bt.slots;
    const uint64_t wait_ns = bt.job[0].wait_ns;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSA; s++) {
            tc::mbar_init(&fullA[s], 1);
            tc::mbar_init(&emptyA[s], 8);
        }
        for (int s = 0; s < 3 * kSB; s++) {
            tc::mbar_init(&fullB[s], 1);
            tc::mbar_init(&emptyB[s], kGauss ? 1 : 2);
        }
        for (int s = 0; s < kBars; s++) {
            tc::mbar_init(&aFull[s], kH == 1 ? 8 : 4);
            tc::mbar_init(&aEmpty[s], kGauss ? 1 : 2);
        }
        for (int t = 0; t < 3; t++) tc::mbar_init(&accFull[t], 1);
        for (uint32_t t = 0; t < AccState::kEnds; t++) tc::mbar_init(&accEmpty[t], kDrainWarps);
        tc::mbar_init(&mmaDone, kP);
        abort_flag = 0;
        tc::mbar_fence_init();
    }
    if (warp == 1) tc::tmem_alloc(&tmem_base, kTmemCols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_base;
    follow();

    struct Unit {
        int jb, x, y, z, m, c0, c1;
    };
    auto unit = [&](int u) {
        Unit n;
        n.jb = 0;
        while (n.jb + 1 < bt.njobs && u >= bt.job[n.jb + 1].unit0) n.jb++;
        const RsJob &a = bt.job[n.jb];
        int r = u - a.unit0;
        n.x = r % a.tx;
        r /= a.tx;
        n.y = r % a.ty;
        r /= a.ty;
        n.z = r % a.tz;
        n.m = r / a.tz;
        n.c0 = n.z * a.cs;
        n.c1 = min(a.nch, n.c0 + a.cs);
        return n;
    };

    // A wait of a whole warp: every lane waits (bounded), and all leave with
    // the same answer, so that no lane is missed at the next warp barrier.
    auto wait_all = [&](uint32_t b, uint32_t parity) {
        const bool r = tc::mbar_wait_at(b, parity, &abort_flag, wait_ns);
        return __all_sync(0xffffffffu, r) != 0;
    };
    const uint32_t aF = tc::smem_u32(aFull), aE = tc::smem_u32(aEmpty);
    const uint32_t bars = aF;                      // aligned to its size: a stage's barrier by or-ing
    constexpr uint32_t kBarMask = 8 * kBars - 1, kBarEmpty = 8 * kBars;

    int fills = 0;      // copies issued, of A (warp 0) or B (warps 1-3, or warp 3)
    if (warp < 4) {
      if (Cfg::kR0) tc::reg_dec<Cfg::kR0 ? Cfg::kR0 : 24>();
      if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
                const Unit n = unit(u);
                const RsJob &a = bt.job[n.jb];
                const uint8_t *src = a.A + (((int64_t)n.m * a.ty + n.y) * a.nch + n.c0) * kAStage;
                for (int c = n.c0; c < n.c1; c++, src += kAStage) {
                    const int s = fills % kSA, f = fills / kSA;
                    if (f >= 1 && !tc::mbar_wait(&emptyA[s], (f - 1) & 1, &abort_flag, wait_ns)) { ok = false; break; }
                    tc::mbar_expect_tx(&fullA[s], kAStage);
                    tc::bulk_load(sA + s * kAStage, src, kAStage, &fullA[s]);
                    fills++;
                }
            }
        }
      } else if constexpr (kGauss) {
        // A warp for each product: its waits and instructions are a third (one
        // warp for all three needed 1.5 to 2 times the MMAs' own time, measured).
        // The whole warp runs the loop and one elected lane issues (predicated,
        // without branches), so that the descriptors are warp-uniform (uniform
        // registers feed tcgen05.mma).  The next chunk's barriers are looked at
        // (without blocking) before this one's MMAs are issued, and waited for
        // only if that look failed.
        const int t = warp - 1;
        const uint32_t one = tc::elect_one() ? 1u : 0u;
        const uint32_t fullB0 = tc::smem_u32(fullB + t * kSB), emptyB0 = tc::smem_u32(emptyB + t * kSB);
        const uint32_t accF = tc::smem_u32(&accFull[t]), accE = tc::smem_u32(&accEmpty[t]);
        const uint32_t acc = tmem + t * stride, tbeg = tmem + 3 * stride, tend = tbeg + slots * kCols;
        bool ok = true;
        uint32_t sB8 = 0, sph = 0, aph = 1;        // stage of B (8 bytes a barrier), phases
        // The warp also copies its part of B (a third of the stage whatever the width:
        // the products' warps reuse a stage independently of one another), kSB - 1 chunks ahead: into the stage
        // whose MMAs it issued a chunk ago (one thread that copied A and all of B
        // spent up to 1650 cycles a chunk on it, measured, more than any other role).
        int uL = blockIdx.x, leftL = 0, xL = 0, zL = 0;
        const CUtensorMap *mapL = nullptr;
        uint32_t bytesL = 0;
        const uint32_t sB0 = tc::smem_u32(sB) + t * (kBStage / 3);
        uint32_t l8 = 0, lph = 1;
        bool rdyE = false;                         // its stage was seen free
        auto load = [&]() {
            if (leftL == 0) {
                if (uL >= units) return true;
                const Unit n = unit(uL);
                const RsJob &a = bt.job[n.jb];
                mapL = &a.tmB;
                bytesL = (uint32_t)a.w * kChunk * 2;
                xL = n.x * a.w;
                zL = (n.m * a.nch + n.c0) * 3 + t;
                leftL = n.c1 - n.c0;
                uL += gridDim.x;
            }
            if (!rdyE && !wait_all(emptyB0 + l8, lph)) return false;
            tc::tma_load_3d_if(one, sB0 + l8 * (kBStage / 8), mapL, 0, xL, zL, fullB0 + l8, bytesL);
            fills++;
            zL += 3;
            leftL--;
            l8 += 8;
            if (l8 == 8 * kSB) { l8 = 0; lph ^= 1; }
            return true;
        };
        for (int s = 0; s + 1 < kSB; s++) load();   // fresh barriers: no wait
        // The product's stage of a chunk (or half of it), its barrier and phase.  A wait that
        // succeeds costs a warp about 100 cycles, so the barriers of the next
        // stage are looked at (without blocking) before this one's MMAs are issued,
        // and waited for only if that look failed.
        uint32_t f8 = 8 * t, bph = 0, at = tbeg + kCols * t;
        bool rdy = false, rdyB = false;
        auto next = [&]() { return bars | f8; };
        auto advance = [&]() {
            f8 += 24;
            if (f8 > kBarMask) { f8 &= kBarMask; bph ^= 1; }
            at += 3 * kCols;
            if (at >= tend) at -= slots * kCols;
        };
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const Unit n = unit(u);
            const int w = bt.job[n.jb].w;
            const uint32_t id = tc::idesc_f16_f32(kRows, w);
            const uint64_t bd0 = tc::sdesc_sw128(sB) + (uint32_t)(t * (kBStage / 3) >> 4);
            const int nc = n.c1 - n.c0;
            uint32_t fresh = 1;
            for (int c = 0; c < nc; c++) {
                const uint32_t end = c + 1 == nc || range_end(t, c) ? 1u : 0u;
                if (!rdyB && !wait_all(fullB0 + sB8, sph)) { ok = false; break; }
                // a fresh barrier passes the wait for the phase before its first
                if (fresh && !wait_all(accE, aph)) { ok = false; break; }
                const uint64_t bd = bd0 + (uint64_t)(sB8 * (kBStage / 8 >> 4));
                bool lookB = false, lookE = false;
#pragma unroll
                for (int h = 0; h < kH; h++) {
                    const uint32_t b0 = next();
                    if (!rdy && !wait_all(b0, bph)) { ok = false; break; }
                    tc::fence_after();
                    const uint32_t t0 = at, eB = emptyB0 + sB8;
                    advance();
                    const bool look = tc::mbar_test_at(next(), bph);
                    if (h == kH - 1) {
                        sB8 += 8;
                        if (sB8 == 8 * kSB) { sB8 = 0; sph ^= 1; }
                        lookB = tc::mbar_test_at(fullB0 + sB8, sph);
                        lookE = tc::mbar_test_at(emptyB0 + l8, lph);
                    }
#pragma unroll
                    for (int k = 0; k < 4 / kH; k++)
                        tc::mma_f16_ta_if(one, acc, t0 + 8 * k, bd + 2 * (h * (4 / kH) + k), id,
                                          h + k == 0 ? fresh ^ 1 : 1u);
                    tc::mma_commit_if(one, b0 + kBarEmpty);
                    if (h == kH - 1) {
                        tc::mma_commit_if(one, eB);
                        if (end) tc::mma_commit_if(one, accF);
                    }
                    rdy = __all_sync(0xffffffffu, look) != 0;
                }
                if (!ok) break;
                fresh = end;
                aph ^= end;
                rdyB = __all_sync(0xffffffffu, lookB) != 0;
                rdyE = __all_sync(0xffffffffu, lookE) != 0;
                if (!load()) { ok = false; break; }
            }
        }
      } else if (warp == 3) {
        if (lane == 0) {
            bool ok = true;
            for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
                const Unit n = unit(u);
                const RsJob &a = bt.job[n.jb];
                const uint32_t bytes = (uint32_t)a.w * kChunk * 2 * 2;
                const int x = n.x * a.w;
                int z = (n.m * a.nch + n.c0) * 2;
                for (int c = n.c0; c < n.c1; c++, z += 2) {
                    const int s = fills % kSB, f = fills / kSB;
                    if (f >= 1 && !tc::mbar_wait(&emptyB[s], (f - 1) & 1, &abort_flag, wait_ns)) { ok = false; break; }
                    tc::mbar_expect_tx(&fullB[s], bytes);
                    tc::tma_load_3d(sB + s * kBStage, &a.tmB, 0, x, z, &fullB[s]);
                    fills++;
                }
            }
        }
      } else {
        // A warp for each accumulator.  The whole warp runs the loop and one elected
        // lane issues (predicated, without branches), so that the descriptors are
        // warp-uniform (uniform registers feed tcgen05.mma).  A wait that succeeds
        // costs a warp about 100 cycles, so the barriers of the next stage are
        // looked at (without blocking) before this one's MMAs are issued, and waited
        // for only if that look failed.
        const int t = warp - 1;
        const uint32_t one = tc::elect_one() ? 1u : 0u;
        const uint32_t fB = tc::smem_u32(fullB), eB = tc::smem_u32(emptyB);
        const uint32_t accF = tc::smem_u32(accFull), accE = tc::smem_u32(accEmpty);
        const uint32_t tbeg = tmem + 3 * stride, s8end = slots * 8;
        bool ok = true, rdy = false, rdyB = false;
        uint32_t sB8 = 0, sph = 0;                 // stage of B (8 bytes a barrier), phase
        AccState st;
        uint32_t s8 = 0, bph = 0, at = tbeg;       // stage of A
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const Unit n = unit(u);
            const int w = bt.job[n.jb].w;
            const uint32_t id = tc::idesc_f16_f32(kRows, w), id2 = t == 0 ? id | tc::kIdescNegA : id;
            const uint64_t part = (uint64_t)(w * kChunk * 2 >> 4);
            const uint64_t bd1 = tc::sdesc_sw128(sB) + (t == 0 ? 0 : part), bd2 = tc::sdesc_sw128(sB) + (t == 0 ? part : 0);
            const int nc = n.c1 - n.c0;
            uint32_t fresh = 1;
            for (int c = 0; c < nc; c++) {
                const int dr = drained_after(c, nc);
                const uint32_t end = c + 1 == nc || dr == t ? 1u : 0u, buf = t == 0 ? st.b[0] : st.b[1];
                const uint32_t acc = tmem + buf * stride;
                if (!rdyB && !wait_all(fB + sB8, sph)) { ok = false; break; }
                // a fresh barrier passes the wait for the phase before its first
                if (fresh && !wait_all(accE + 8 * st.wait_on(buf), st.wait_parity(buf))) { ok = false; break; }
                const uint64_t bo = (uint64_t)(sB8 * (kBStage / 8 >> 4));
                const uint32_t eb = eB + sB8;
                bool lookB = false;
#pragma unroll
                for (int h = 0; h < kH; h++) {
                    if (!rdy && !wait_all(aF + s8, bph)) { ok = false; break; }
                    tc::fence_after();
                    const uint32_t t0 = at, e0 = aE + s8;
                    at += kCols;
                    s8 += 8;
                    if (s8 == s8end) { s8 = 0; bph ^= 1; at = tbeg; }
                    const bool look = tc::mbar_test_at(aF + s8, bph);
                    if (h == kH - 1) {
                        sB8 += 8;
                        if (sB8 == 8 * kSB) { sB8 = 0; sph ^= 1; }
                        lookB = tc::mbar_test_at(fB + sB8, sph);
                    }
#pragma unroll
                    for (int k = 0; k < 4 / kH; k++) {
                        const uint64_t ko = bo + 2 * (h * (4 / kH) + k);
                        tc::mma_f16_ta_if(one, acc, t0 + 8 * k, bd1 + ko, id, h + k == 0 ? fresh ^ 1 : 1u);
                        tc::mma_f16_ta_if(one, acc, t0 + kCols / 2 + 8 * k, bd2 + ko, id2, 1u);
                    }
                    tc::mma_commit_if(one, e0);
                    if (h == kH - 1) {
                        tc::mma_commit_if(one, eb);
                        if (end) tc::mma_commit_if(one, accF + 8 * buf);
                    }
                    rdy = __all_sync(0xffffffffu, look) != 0;
                }
                if (!ok) break;
                fresh = end;
                if (dr >= 0) st.end(dr);
                rdyB = __all_sync(0xffffffffu, lookB) != 0;
            }
            st.end(0);
            st.end(1);
        }
      }
    } else if (warp < 4 + kConvWarps) {
        if (Cfg::kRC) tc::reg_dec<Cfg::kRC ? Cfg::kRC : 24>();
        // The groups take turns, half a chunk (32 K elements) each: item 2 chunk + h,
        // which is a stage, or with kH = 1 its half h.  Gauss: its i-th operand is fill
        // 3 item + i of the ring of stages, and waits for the MMAs on the fill `slots`
        // before it.
        const int quad = warp & 3, row = quad * 32 + lane;
        const __half2 k1152 = __floats2half2_rn(1152.f, 1152.f);
        int item = (warp - 4) >> 2;
        uint32_t s = kH == 1 ? item >> 1 : item, ph = 1;   // its stage; phase of the wait for it
        const uint32_t tbeg = tmem + ((uint32_t)(quad * 32) << 16) + 3 * stride, tend = tbeg + slots * kCols;
        uint32_t f8 = 24 * item;                   // Gauss: the fill's barrier
        uint32_t e8 = 8 * (3 * item - slots), eph = (int)e8 >= 0 ? 0 : 1;   // of the fill it waits for (modulo the ring)
        e8 &= kBarMask;
        uint32_t ta = tbeg + 3 * item % slots * kCols;
        uint32_t sa8 = 8 * (item >> 1), saph = 0;  // stage of A's bytes (8 bytes a barrier), and its phase
        const uint32_t fullA0 = tc::smem_u32(fullA), emptyA0 = tc::smem_u32(emptyA);
        auto convert = [&](const uint8_t *src, uint32_t *r) {
#pragma unroll
            for (int g = 0; g < 2; g++) {
                const uint4 q = *(const uint4 *)(src + g * (kRows * 16));
                const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    const uint32_t x = __byte_perm(v[e / 2], 0x64646464u, e % 2 ? 0x4342 : 0x4140);
                    __half2 a;                     // (1024 + b) - 1152
                    memcpy(&a, &x, 4);
                    a = __hsub2(a, k1152);
                    memcpy(&r[g * 8 + e], &a, 4);
                }
            }
        };
        // Gauss: store an operand's columns and tell its product's MMAs
        auto put = [&](const uint32_t *r) {
            // a fresh barrier passes the wait for the phase before its first
            if (!wait_all(bars | kBarEmpty | e8, eph)) return false;
            tc::fence_after();
            tc::tmem_st16(ta, r);
            ta += kCols;
            if (ta == tend) ta = tbeg;
            e8 += 8;
            if (e8 > kBarMask) { e8 = 0; eph ^= 1; }
            tc::tmem_wait_st();
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive_at(bars | f8);
            f8 = (f8 + 8) & kBarMask;
            return true;
        };
        // item counts over all units; i is its number in its unit
        int done = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const Unit n = unit(u);
            const int ni = 2 * (n.c1 - n.c0);
            for (int i = item - done; i < ni; i += kConvGroups, item += kConvGroups) {
                if (!wait_all(fullA0 + sa8, saph)) { ok = false; break; }
                const int h = i & 1;
                const uint8_t *src = sA + sa8 * (kAStage / 8) + (h * 2 * kRows + row) * 16;
                uint32_t re[16], im[16];           // FP16 pairs
                convert(src, re);
                convert(src + 4 * kRows * 16, im);
                __syncwarp();
                if (lane == 0) tc::mbar_arrive_at(emptyA0 + sa8);
                const int chunks = (h + kConvGroups) / 2;
                if constexpr (kGauss) {
                    if (!put(re) || !put(im)) { ok = false; break; }
#pragma unroll
                    for (int e = 0; e < 16; e++) {
                        __half2 a, b;
                        memcpy(&a, &re[e], 4);
                        memcpy(&b, &im[e], 4);
                        a = __hadd2(a, b);         // in [-256, 254]: exact
                        memcpy(&re[e], &a, 4);
                    }
                    if (!put(re)) { ok = false; break; }
                    // past the other groups' items
                    constexpr uint32_t over = 3 * (kConvGroups - 1);
                    f8 = (f8 + 8 * over) & kBarMask;
                    e8 += 8 * over;
                    if (e8 > kBarMask) { e8 &= kBarMask; eph ^= 1; }
                    ta += over * kCols;            // at most one turn of the ring
                    if (ta >= tend) ta -= slots * kCols;
                } else {
                    // a fresh barrier passes the wait for the phase before its first
                    if (!wait_all(aE + 8 * s, ph)) { ok = false; break; }
                    tc::fence_after();
                    const uint32_t at = tbeg + s * kCols + (kH == 1 ? 16 * h : 0);
                    tc::tmem_st16(at, re);
                    tc::tmem_st16(at + kCols / 2, im);
                    tc::tmem_wait_st();
                    tc::fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive_at(aF + 8 * s);
                    s += kH == 1 ? chunks : kConvGroups;
                    if (s >= slots) { s -= slots; ph ^= 1; }
                }
                sa8 += chunks * 8;
                if (sa8 >= 8 * kSA) { sa8 -= 8 * kSA; saph ^= 1; }
            }
            done += ni;
        }
    } else {
        if (Cfg::kRD) tc::reg_inc<Cfg::kRD ? Cfg::kRD : 24>();
        const int quad = warp & 3, half = (warp - 4 - kConvWarps) >> 2;
        const int row = quad * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        constexpr int kG = Cfg::kW / 16, kHold = Cfg::kHold;   // granules of 8 columns per thread, held at once
        constexpr float kMagic = 12582912.f;       // 1.5 2^23: rounds to an integer
        bool ok = true;
        AccState st;
        uint32_t gph = 0;                          // Gauss: phases of accFull
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const Unit n = unit(u);
            const RsJob &a = bt.job[n.jb];
            const int ng = a.w / 16;
            const float pf = kTab.m[n.m].pf, inv = kTab.m[n.m].inv;
            int acc[kG * 8];
#pragma unroll
            for (int v = 0; v < kG * 8; v++) acc[v] = 0;
            int cnt = 0;
            const int nc = n.c1 - n.c0;
            const uint64_t inv2 = tc::pin2(tc::f32x2(inv, inv)), mp2 = tc::pin2(tc::f32x2(-pf, -pf));
            const uint64_t magic2 = tc::pin2(tc::f32x2(kMagic, kMagic)), mmagic2 = tc::pin2(tc::f32x2(-kMagic, -kMagic));
            for (int ev = 0, fin = 0; fin < kP;) {
                int t;
                uint32_t buf, phase, done;
                float coef;                        // Re + kPack Im
                if constexpr (kGauss) {
                    // T2, T1, T2, T0 after chunks 5, 10, 13, 15 of every 16, until the
                    // last chunk; then T0, T1, T2
                    if (fin == 0 && (ev >> 2) * 16 + ((0xFDA5 >> (ev % 4 * 4)) & 15) < nc - 1) {
                        t = (0x0212 >> (ev % 4 * 4)) & 3;
                        ev++;
                    } else {
                        t = fin++;
                    }
                    buf = done = (uint32_t)t;
                    phase = gph >> t & 1;
                    gph ^= 1u << t;
                    // T0 counts (1, -1), T1 (-1, -1), T2 (0, 1)
                    coef = t == 0 ? (float)(1 - kPack) : t == 1 ? (float)(-1 - kPack) : (float)kPack;
                } else {
                    // Im and Re by turns after every fourth chunk, until the last
                    // chunk; then Re, Im
                    t = fin == 0 ? drained_after(4 * ev + 3, nc) : -1;
                    if (t >= 0) ev++;
                    else t = fin++;
                    buf = t == 0 ? st.b[0] : st.b[1];
                    phase = st.drains >> buf & 1;
                    done = st.signal();
                    st.end(t);
                    coef = t == 0 ? 1.f : (float)kPack;
                }
                if (!wait_all(tc::smem_u32(&accFull[buf]), phase)) { ok = false; break; }
                tc::fence_after();
                const uint64_t coef2 = tc::pin2(tc::f32x2(coef, coef));
                const uint32_t col = tmem + lane_addr + buf * stride + half * ng * 8;
                auto digest = [&](const uint32_t *r, int g) {
#pragma unroll
                    for (int v = 0; v < 8; v += 2) {
                        const uint64_t xx = tc::pack2(r[v], r[v + 1]);
                        const uint64_t q = tc::add2(tc::fma2(xx, inv2, magic2), mmagic2);
                        const uint64_t y = tc::fma2(q, mp2, xx);
                        const uint64_t z = tc::fma2(y, coef2, magic2);
                        acc[g * 8 + v] += (int)(uint32_t)z;
                        acc[g * 8 + v + 1] += (int)(uint32_t)(z >> 32);
                    }
                };
                // as many columns as registers hold are loaded first, then the
                // accumulator goes back to the MMAs, then the arithmetic
                uint32_t r[kHold * 8];
#pragma unroll
                for (int g = 0; g < kHold; g++)
                    if (g < ng) tc::tmem_ld8(col + g * 8, r + g * 8);
                tc::tmem_wait_ld();
#pragma unroll
                for (int g = kHold; g < kG; g++)
                    if (g < ng) {
                        digest(r + (g - kHold) * 8, g - kHold);
                        tc::tmem_ld8(col + g * 8, r + (g - kHold) * 8);
                    }
                tc::tmem_wait_ld();
                tc::fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&accEmpty[done]);
#pragma unroll
                for (int g = 0; g < kG; g++) {
                    const int at = g >= kHold ? g - kHold : g;
                    if (g < ng && (g >= kG - kHold || g + kHold >= ng)) digest(r + at * 8, g);
                }
                cnt++;
            }
            if (!ok) break;
            uchar2 *R = a.R + ((int64_t)(n.m * a.tz + n.z) * a.mp + n.x * a.w + half * ng * 8) * a.Mp +
                       (int64_t)n.y * kRows + row;
            const unsigned off = (unsigned)cnt * (unsigned)__float_as_int(kMagic);
            const uint64_t byte2 = tc::pin2(tc::f32x2(8388736.f, 8388736.f));
#pragma unroll
            for (int v = 0; v < kG * 8; v++) {
                if (v < ng * 8) {
                    const int s = (int)((unsigned)acc[v] - off);
                    const int si = (s + kPack / 2) >> 13, sr = s - si * kPack;
                    // to FP32 and back by the bit patterns of 1.5 2^23 + x and 2^23 + 128 + r
                    const uint64_t xx = tc::add2(tc::pack2(0x4B400000u + (uint32_t)sr, 0x4B400000u + (uint32_t)si), mmagic2);
                    const uint64_t q = tc::add2(tc::fma2(xx, inv2, magic2), mmagic2);
                    const uint64_t z = tc::add2(tc::fma2(q, mp2, xx), byte2);
                    R[(int64_t)v * a.Mp] = make_uchar2((uint8_t)z, (uint8_t)(z >> 32));
                }
            }
        }
    }

    tc::fence_before();
    __syncthreads();
    if (abort_flag) {
        // An expired wait: every role has left its loop.  Before shared and
        // tensor memory go, the copies and MMAs already issued must land.
        bool drained = true;
        if (warp == 0 && lane == 0) {
            for (int s = 0; s < kSA; s++) {
                const int f = (fills - s + kSA - 1) / kSA;           // copies into stage s
                if (f > 0) drained &= tc::mbar_wait_for(&fullA[s], (f - 1) & 1, kWindDownNs);
            }
        }
        if (kGauss ? warp >= 1 && warp < 4 : warp == 3) {
            // lane 0 knows the copies issued: alone with four products, with
            // Gauss every lane counts them
            if (lane == 0)
                for (int s = 0; s < kSB; s++) {
                    const int f = (fills - s + kSB - 1) / kSB;
                    if (f > 0)
                        drained &= tc::mbar_wait_for(&fullB[(kGauss ? (warp - 1) * kSB : 0) + s], (f - 1) & 1, kWindDownNs);
                }
        }
        if (warp >= 1 && warp <= kP && tc::elect_one()) {
            tc::mma_commit(&mmaDone);
            drained &= tc::mbar_wait_for(&mmaDone, 0, kWindDownNs);
        }
        if (!drained)
            for (int j = 0; j < bt.njobs; j++) set_error(bt.job[j].sc, DEV_TIMEOUT, -1 - (int)blockIdx.x);
        tc::fence_before();
        __syncthreads();
        if (threadIdx.x == 0)
            for (int j = 0; j < bt.njobs; j++) set_error(bt.job[j].sc, DEV_TIMEOUT, blockIdx.x);
    }
    if (warp == 1) {
        tc::fence_after();
        tc::tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------ line norms
// The 2-norm of a line (row of A, column of B) only sets a power of two, so
// it is summed in FP32 on the top 20 mantissa bits relative to the largest
// exponent seen, from the bit patterns with integer operations (FP64 issue is
// scarce on this part).  acc 2^(2 (eb - 1023)): the sum of squares, less a
// relative 2^-12 that exponent() adds back.  A subnormal entry may have all its bits
// in the low word: a line without a normal entry (eb 0) is summed once more, by
// add_small.  (With a look at every entry's low word: a product at N = 10008 1669 us
// for 1625.)
struct NormAcc {
    float acc = 0.f;
    int eb = 0;         // biased exponent of the largest entry
    __device__ __forceinline__ void shift_to(int e) {
        const int d = 2 * (e - eb);
        acc = d > 120 ? 0.f : acc * __int_as_float((127 - d) << 23);
        eb = e;
    }
    __device__ __forceinline__ float mant(unsigned h) const {
        const int t = (int)h - ((eb - 127) << 20);
        return (h == 0 || t < 0) ? 0.f : __int_as_float(t << 3);
    }
    __device__ __forceinline__ void add(z_t v) {
        const unsigned hx = (unsigned)__double2hiint(v.x) & 0x7FFFFFFFu;
        const unsigned hy = (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu;
        const int e = (int)(max(hx, hy) >> 20);
        if (e > eb) shift_to(e);
        const float fx = mant(hx), fy = mant(hy);
        acc = fmaf(fx, fx, fmaf(fy, fy, acc));
    }
    // |x| 2^1023 of zero and subnormal x; eb stays 0
    static __device__ __forceinline__ float small(double x) {
        return (float)((unsigned long long)__double_as_longlong(x) & 0xFFFFFFFFFFFFFull) * 0x1.0p-51f;
    }
    __device__ __forceinline__ void add_small(z_t v) {
        const float fx = small(v.x), fy = small(v.y);
        acc = fmaf(fx, fx, fmaf(fy, fy, acc));
    }
    __device__ __forceinline__ void add(float2 o) { merge(o.x, __float_as_int(o.y)); }
    __device__ __forceinline__ void merge(float oacc, int oeb) {
        if (oeb > eb) shift_to(oeb);
        const int d = 2 * (eb - oeb);
        if (d <= 120) acc = fmaf(oacc, __int_as_float((127 - d) << 23), acc);
    }
    __device__ __forceinline__ float2 pack() const { return make_float2(acc, __int_as_float(eb)); }
    // h with norm <= 2^h; INT_MIN for a zero line
    __device__ __forceinline__ int exponent() const {
        if (!(acc > 0.f)) return INT_MIN;
        int e;
        frexpf(acc * (1.f + 0x1.0p-10f), &e);
        return (e + 2 * (eb - 1023) + 1) >> 1;
    }
};
constexpr int kInfExp = 0x7FF;      // biased exponent of Inf and NaN

// Row sums of squares of the columns [k0, k0 + cols) of A (M rows): one
// partial per row and segment of `seg` columns, partial index seg0 + segment.
__global__ void __launch_bounds__(128)
k_res_rownorm(int64_t M, int64_t cols, const z_t *__restrict__ A, int64_t lda, int seg, int64_t seg0,
              float2 *__restrict__ part) {
    const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (i >= M) return;
    const int64_t k0 = (int64_t)blockIdx.y * seg, k1 = min(k0 + seg, cols);
    NormAcc n;
#pragma unroll 8
    for (int64_t k = k0; k < k1; k++) n.add(A[i + k * lda]);
    if (n.eb == 0) {
        n.acc = 0.f;
        for (int64_t k = k0; k < k1; k++) n.add_small(A[i + k * lda]);
    }
    part[(seg0 + blockIdx.y) * M + i] = n.pack();
}

__global__ void __launch_bounds__(128)
k_res_rowscale(int64_t M, int64_t Mp, int nseg, const float2 *__restrict__ part, int *E, ChaseScalars *sc) {
    const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (i >= Mp) return;
    NormAcc n;
    if (i < M) {
#pragma unroll 8
        for (int s = 0; s < nseg; s++) n.add(part[(int64_t)s * M + i]);
    }
    if (n.eb == kInfExp) set_error(sc, DEV_NONFINITE, (int)i);
    E[i] = n.exponent();
}

// The exponents of all rows in one launch, for up to kSmallSegs segments: 8
// rows a block, a thread per row and segment, and the same sums in the same
// order as the two kernels above.  For short segments only (N < 4096): 17 us
// against 16 + 14 at N = 2000, but with one block for 8 whole rows 1056 us
// against 940 + 17 at N = 20000.  Segments of 8 columns up to N = 1024 fill the
// threads there: a product with its preparation at N = 256 47 -> 40 us (13 moduli; 42 with 14).
// With 32 rows and 8 segments at a time: the rows of a tall A of at most
// kMaxTallCols columns (the general products).
constexpr int kSmallSegs = 128, kMaxTallCols = 512, kTallSegs = kMaxTallCols / 32;
template <int kRowsBlock, int kSegThreads, int kSegs>
__global__ void __launch_bounds__(kRowsBlock *kSegThreads)
k_res_rowexp(int64_t M, int64_t Mp, int64_t K, const z_t *__restrict__ A, int64_t lda, int seg, int nseg, int *E,
             ChaseScalars *sc) {
    __shared__ float2 part[kSegs][kRowsBlock];
    follow();
    const int row = threadIdx.x % kRowsBlock;
    const int64_t i = (int64_t)blockIdx.x * kRowsBlock + row;
    for (int s = threadIdx.x / kRowsBlock; s < nseg; s += kSegThreads) {
        const int64_t k0 = (int64_t)s * seg, k1 = min(k0 + seg, K);
        NormAcc n;
        if (i < M) {
#pragma unroll 8
            for (int64_t k = k0; k < k1; k++) n.add(A[i + k * lda]);
            if (n.eb == 0) {
                n.acc = 0.f;
                for (int64_t k = k0; k < k1; k++) n.add_small(A[i + k * lda]);
            }
        }
        part[s][row] = n.pack();
    }
    __syncthreads();
    if (threadIdx.x >= kRowsBlock || i >= Mp) return;
    NormAcc n;
    if (i < M)
        for (int s = 0; s < nseg; s++) n.add(part[s][row]);
    if (n.eb == kInfExp) set_error(sc, DEV_NONFINITE, (int)i);
    E[i] = n.exponent();
}

// Sum of squares of one column over the block (all threads get it).
template <int kWarps>
__device__ __forceinline__ NormAcc block_norm(NormAcc n, float2 *red) {
    for (int o = 16; o > 0; o >>= 1) {
        const float oa = __shfl_xor_sync(0xffffffffu, n.acc, o);
        const int oe = __shfl_xor_sync(0xffffffffu, n.eb, o);
        n.merge(oa, oe);
    }
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = n.pack();
    __syncthreads();
    NormAcc t;
    for (int w = 0; w < kWarps; w++) t.add(red[w]);
    return t;
}

// Partial sums of squares of column blockIdx.y: part[j * gridDim.x + block]
__global__ void __launch_bounds__(256)
k_res_colnorm(int64_t N, const z_t *__restrict__ Y, int64_t ldy, float2 *__restrict__ part, ChaseScalars *sc) {
    __shared__ float2 red[8];
    follow();
    const int j = blockIdx.y;
    NormAcc n;
    for (int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x; k < N; k += (int64_t)gridDim.x * 256)
        n.add(Y[k + j * ldy]);
    if (n.eb == 0) {
        n.acc = 0.f;
        for (int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x; k < N; k += (int64_t)gridDim.x * 256)
            n.add_small(Y[k + j * ldy]);
    }
    const NormAcc t = block_norm<8>(n, red);
    if (threadIdx.x == 0) {
        if (t.eb == kInfExp) set_error(sc, DEV_NONFINITE, j);
        part[(int64_t)j * gridDim.x + blockIdx.x] = t.pack();
    }
}

// ------------------------------------------------------------ residues
// rint(x 2^sh) + 2^63, ties to even, for |x 2^sh| < 2^62, from the bit
// pattern with integer operations.  Non-finite x gives an arbitrary value.
__device__ __forceinline__ unsigned long long biased_rint(double x, int sh) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7FF);
    unsigned long long m = b & 0xFFFFFFFFFFFFFull;
    int s = -1074 + sh;
    if (ef != 0) {
        m |= 1ull << 52;
        s = ef - 1075 + sh;
    }
    unsigned long long q;
    if (s >= 0) {
        q = m << min(s, 63);
    } else {
        // add half an ulp less one, plus the quotient's last bit: ties to even
        const int r = min(-s, 62);
        const unsigned long long half = 1ull << (r - 1);
        q = (m + half - 1 + ((m >> r) & 1)) >> r;
    }
    q = (b >> 63) ? 0ull - q : q;
    return q + (1ull << 63);
}

// The residues of x0 and x1: words whose low bytes are residue + 128.
struct ResConst {
    uint32_t clo, chi, k0;
    uint64_t mp2, inv2;
    __device__ __forceinline__ explicit ResConst(const ModConst &m)
        : clo(m.clo), chi(m.chi), k0(m.k0), mp2(tc::f32x2(-m.pf, -m.pf)), inv2(tc::f32x2(m.inv, m.inv)) {}
    __device__ __forceinline__ uint64_t two(unsigned long long x0, unsigned long long x1) const {
        const uint64_t magic2 = tc::f32x2(12582912.f, 12582912.f), mmagic2 = tc::f32x2(-12582912.f, -12582912.f);
        const uint64_t bias2 = tc::f32x2(8388736.f, 8388736.f);
        const uint32_t v0 = __dp4a((uint32_t)(x0 >> 32), chi, __dp4a((uint32_t)x0, clo, k0));
        const uint32_t v1 = __dp4a((uint32_t)(x1 >> 32), chi, __dp4a((uint32_t)x1, clo, k0));
        const uint64_t f = tc::pack2(v0, v1);
        const uint64_t q = tc::add2(tc::fma2(f, inv2, magic2), mmagic2);
        return tc::add2(tc::fma2(q, mp2, f), bias2);
    }
};

// The residues of EL consecutive K elements of a row: EL bytes of Re, and of Im
// half a chunk's block on, for each modulus mstep apart.
template <int EL>
__device__ __forceinline__ void residues_of_row(const z_t *v, int sh, int nmod, int64_t mstep, uint8_t *dst) {
#pragma unroll
    for (int part = 0; part < 2; part++) {
        unsigned long long x[EL];
#pragma unroll
        for (int e = 0; e < EL; e++) x[e] = biased_rint(part ? v[e].y : v[e].x, sh);
        uint8_t *d = dst + part * (4 * kRows * 16);
#pragma unroll 1
        for (int m = 0; m < nmod; m++, d += mstep) {
            const ResConst rc(kTab.m[m]);
            uint32_t o[EL / 4];
#pragma unroll
            for (int q = 0; q < EL / 4; q++) {
                const uint64_t a = rc.two(x[q * 4], x[q * 4 + 1]), b = rc.two(x[q * 4 + 2], x[q * 4 + 3]);
                const uint32_t lo = __byte_perm((uint32_t)a, (uint32_t)(a >> 32), 0x0040);
                const uint32_t hi = __byte_perm((uint32_t)b, (uint32_t)(b >> 32), 0x0040);
                o[q] = __byte_perm(lo, hi, 0x5410);
            }
            if (EL == 16) *(uint4 *)d = make_uint4(o[0], o[EL / 16], o[EL / 8], o[EL / 16 * 3]);
            else *(uint32_t *)d = o[0];
        }
    }
}

// Residues of 16 consecutive K elements of one row of A per thread: columns
// k0 + 16 (blockIdx.x) of the matrix, read coalesced down the rows, and for
// each modulus 16 bytes of Re and of Im, [group of 16][row][16 bytes] of the
// chunk's 16 KB block, so that a converter thread's row is conflict-free.
// Bound by integer issue: about 140 instructions per element for the 28
// residues, over 16 bytes read and 28 written.
template <int EL>   // K elements of a thread: 16, or 4 to fill the SMs from a small matrix
__global__ void __launch_bounds__(128, 4)
k_res_slice_a(int64_t M, int64_t K, const z_t *__restrict__ A, int64_t lda, int64_t kbase, int64_t T,
              int64_t nch, const int *__restrict__ E, int nmod, int bits, uint8_t *__restrict__ S) {
    follow();
    const int row = threadIdx.x;
    const int64_t i = (int64_t)blockIdx.y * kRows + row;
    const int64_t k0 = (int64_t)blockIdx.x * EL;               // within this panel
    const int64_t kg = kbase + k0;                             // of the whole matrix
    int sh = 0;
    bool live = i < M;
    if (live) {
        const int e = E[i];
        live = e != INT_MIN;
        sh = live ? bits - e : 0;
    }
    z_t v[EL];
#pragma unroll
    for (int e = 0; e < EL; e++) v[e] = (live && kg + e < K) ? A[i + (k0 + e) * lda] : zmk(0.0, 0.0);
    const int64_t c = kg / kChunk;
    const int g = (int)(kg % kChunk) / 16;
    uint8_t *dst = S + ((int64_t)blockIdx.y * nch + c) * kAStage + g * (kRows * 16) + row * 16 + (int)(kg % 16);
    residues_of_row<EL>(v, sh, nmod, T * nch * kAStage, dst);
}

// The same of A^H for A with long columns (K x M): 32 columns by 64 elements a
// block, read along the columns and turned in shared memory.  E[i] receives
// column i's exponent, from its partial sums of squares.  K = 20000, 100 columns:
// 46 us, 32 MB read and 60 written.
__global__ void __launch_bounds__(128, 4)
k_res_slice_ah(int64_t M, int64_t K, const z_t *__restrict__ A, int64_t lda, int64_t T, int64_t nch, int npart,
               const float2 *__restrict__ part, int *__restrict__ E, int nmod, int bits, uint8_t *__restrict__ S) {
    __shared__ z_t tile[32][kChunk + 1];
    follow();
    const int64_t i0 = (int64_t)blockIdx.y * 32, c = blockIdx.x;
    for (int e = threadIdx.x; e < 32 * kChunk; e += 128) {
        const int64_t k = c * kChunk + e % kChunk, i = i0 + e / kChunk;
        tile[e / kChunk][e % kChunk] = (k < K && i < M) ? A[k + i * lda] : zmk(0.0, 0.0);
    }
    const int r = threadIdx.x % 32, g = threadIdx.x / 32;
    const int64_t i = i0 + r;
    NormAcc n;
    if (i < M)
        for (int s = 0; s < npart; s++) n.add(part[i * npart + s]);
    const int h = n.exponent();
    if (blockIdx.x == 0 && g == 0 && i < M) E[i] = h;
    __syncthreads();
    z_t v[16];
#pragma unroll
    for (int e = 0; e < 16; e++) {
        const z_t x = tile[r][g * 16 + e];
        v[e] = h != INT_MIN ? zmk(x.x, -x.y) : zmk(0.0, 0.0);
    }
    uint8_t *dst = S + (i / kRows * nch + c) * kAStage + g * (kRows * 16) + (int)(i % kRows) * 16;
    residues_of_row<16>(v, h != INT_MIN ? bits - h : 0, nmod, T * nch * kAStage, dst);
}

// FP16 residues of Y, -> [modulus][chunk][Re, Im, and Re + Im with parts = 3][column][64]: one
// column and 8 consecutive K elements per thread, the moduli from blockIdx.z
// in steps of gridDim.z.  The column's norm comes from its partial sums, or with
// npart = 0 from the column itself; F[j] receives its exponent.
__global__ void __launch_bounds__(128)
k_res_slice_b(int64_t N, int64_t Kp, int n, int mp, const z_t *__restrict__ Y, int64_t ldy, int npart,
              const float2 *__restrict__ part, int *__restrict__ F, int nmod, int bits, int parts,
              uint16_t *__restrict__ B, ChaseScalars *sc) {
    follow();
    const int j = blockIdx.y;
    const int64_t k = ((int64_t)blockIdx.x * 128 + threadIdx.x) * 8;
    int h = INT_MIN;
    if (npart == 0) {                      // a short column: its norm here
        __shared__ float2 red[4];
        NormAcc a;
        if (j < n) {
#pragma unroll 4
            for (int64_t i = threadIdx.x; i < N; i += 128) a.add(Y[i + j * ldy]);
            if (a.eb == 0) {
                a.acc = 0.f;
                for (int64_t i = threadIdx.x; i < N; i += 128) a.add_small(Y[i + j * ldy]);
            }
        }
        a = block_norm<4>(a, red);
        if (a.eb == kInfExp) set_error(sc, DEV_NONFINITE, j);
        h = a.exponent();
    } else if (j < n) {
        NormAcc a;
        for (int s = 0; s < npart; s++) a.add(part[(int64_t)j * npart + s]);
        h = a.exponent();
    }
    if (blockIdx.x == 0 && blockIdx.z == 0 && threadIdx.x == 0) F[j] = h;
    if (k >= Kp) return;
    const bool live = h != INT_MIN;
    const int sh = live ? bits - h : 0;
    unsigned long long xr[8], xi[8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
        const z_t y = (live && k + e < N) ? Y[k + e + j * ldy] : zmk(0.0, 0.0);
        xr[e] = biased_rint(y.x, sh);
        xi[e] = biased_rint(y.y, sh);
    }
    const int64_t nch = Kp / kChunk, c = k / kChunk;
    const int64_t pstep = (int64_t)mp * kChunk;
    const __half2 bias = __floats2half2_rn(1152.f, 1152.f);
#pragma unroll 1
    for (int m = blockIdx.z; m < nmod; m += gridDim.z) {
        const ResConst rc(kTab.m[m]);
        const int p = (int)kTab.m[m].pf;
        uint32_t o[3][4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            // bytes residue + 128 of two elements, 16 bits each: Re, Im, Re + Im
            const uint64_t a = rc.two(xr[q * 2], xr[q * 2 + 1]), b = rc.two(xi[q * 2], xi[q * 2 + 1]);
            const uint32_t wr = __byte_perm((uint32_t)a, (uint32_t)(a >> 32), 0x0400) & 0x00FF00FFu;
            const uint32_t wi = __byte_perm((uint32_t)b, (uint32_t)(b >> 32), 0x0400) & 0x00FF00FFu;
            uint32_t ws = 0;
            if (parts == 3) {
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    // the sum modulo p, in [-128, 127]
                    int s = (int)(wr >> (16 * e) & 255) + (int)(wi >> (16 * e) & 255) - 256;
                    s += s < -128 ? p : 0;
                    s -= s > 127 ? p : 0;
                    ws |= (uint32_t)(s + 128) << (16 * e);
                }
            }
            const uint32_t w[3] = {wr, wi, ws};
#pragma unroll
            for (int t = 0; t < 3; t++) {
                const uint32_t x = 0x64006400u | w[t];
                __half2 hh;
                memcpy(&hh, &x, 4);
                hh = __hsub2(hh, bias);
                memcpy(&o[t][q], &hh, 4);
            }
        }
        uint16_t *d = B + (((int64_t)m * nch + c) * parts) * pstep + (int64_t)j * kChunk + k % kChunk;
#pragma unroll
        for (int t = 0; t < 3; t++)
            if (t < parts) *(uint4 *)(d + t * pstep) = make_uint4(o[t][0], o[t][1], o[t][2], o[t][3]);
    }
}

// One panel of the synthetic Hamiltonian: all rows, columns j0 .. j0 + cols, as
// bse_build_hamiltonian writes them (the element of the lower triangle, or its
// conjugate), column-major with leading dimension N.
constexpr int kPT = 32;
__global__ void __launch_bounds__(256)
k_res_panel(int Nk, int nb, int N, int jbase, int cols, BseModel md, const double *__restrict__ dE,
            const z_t *__restrict__ u, const z_t *__restrict__ a, const double *__restrict__ Kt,
            z_t *__restrict__ H) {
    extern __shared__ z_t gsm[];
    const int R = md.rank_x;
    z_t *sai = gsm, *saj = gsm + kPT * R;
    const int tx = threadIdx.x, ty = threadIdx.y;      // 32 x 8
    const int i0 = blockIdx.x * kPT, j0 = jbase + blockIdx.y * kPT;
    for (int e = ty * kPT + tx; e < kPT * R; e += kPT * 8) {
        const int t = e / R, r = e % R;
        sai[r * kPT + t] = (i0 + t < N) ? a[(int64_t)(i0 + t) * R + r] : zmk(0.0, 0.0);
        saj[r * kPT + t] = (j0 + t < N) ? a[(int64_t)(j0 + t) * R + r] : zmk(0.0, 0.0);
    }
    __syncthreads();
    const int I = i0 + tx;
    if (I >= N) return;
    for (int c = ty; c < kPT; c += 8) {
        const int J = j0 + c;
        if (J >= N || J >= jbase + cols) continue;
        z_t h;
        if (I >= J) h = bse_element(I, J, R, sai + tx, saj + c, kPT, u[I], u[J], dE[I], Nk, nb, md.w0, Kt);
        else h = zconj(bse_element(J, I, R, saj + c, sai + tx, kPT, u[J], u[I], dE[J], Nk, nb, md.w0, Kt));
        H[I + (int64_t)(J - jbase) * N] = h;
    }
}

// ------------------------------------------------------------ the result
// Element (i, j) from the residues of all moduli and splits, ROWS consecutive
// rows per thread (4, or 1 to fill the SMs from a small result).  The splits' bytes (residue + 128) are summed two to a
// word first, then F = sum_m W_m u_m - nz bias, a multiply-add per word of W:
// 14 us at N = 2000, 75 columns, and with four rows a thread 88 us at N = 20000, 140 columns
// (from HBM).  With 13 moduli and 64-bit fractions: 10 us at N = 2000 (15 with four rows per
// thread, and 20 with a 64-bit product per split and value before; 23 with the moduli
// shared out over four warps), 7 us at N = 256 (14); 65 at N = 20000 (82 with the loads
// of two moduli in flight, and the conversion and the scaling on the FP64 pipe).
// m 2^e, m >= 2^62, rounded once
__device__ __forceinline__ double to_double(unsigned long long m, int e, bool neg) {
    if (!(m >> 63)) {
        m <<= 1;
        e--;
    }
    const unsigned long long q = (m >> 11) + (m >> 10 & 1);    // 53 bits, or 2^53
    const int be = e + 63 + 1023;
    double v;
    if (be >= 1 && be <= 2045) v = __longlong_as_double((long long)(((unsigned long long)(be - 1) << 52) + q));
    else v = ldexp((double)m, e);
    return neg ? -v : v;
}
template <int MODS, int BITS, int EXP, unsigned long long MANT, int SET>
struct Recombine {
    static constexpr int kMods = MODS, kWords = 3, kBits = BITS;
    static __device__ __forceinline__ unsigned long long word(int m, int i) { return kTab.m[m].w[SET][i]; }
    // F P 2^(x - 96): |F| P in integers, 64 bits of each, and one rounding to FP64
    // (whose issue is scarce: with conversions and products in FP64 these took longer
    // than the loads)
    static __device__ __forceinline__ double value(const unsigned long long *s, int nz, int x) {
        const unsigned __int128 b = ((unsigned __int128)kTab.bias[SET][1] << 64 | kTab.bias[SET][0]) * (unsigned)nz;
        unsigned __int128 t = s[0] + ((unsigned __int128)s[1] << 32) + ((unsigned __int128)s[2] << 64) - b;
        const bool neg = (uint32_t)(t >> 64) >> 31;            // F: 96 bits, signed
        if (neg) t = 0 - t;
        unsigned long long hi = (unsigned long long)(t >> 32), lo = (unsigned long long)(uint32_t)t << 32;
        int lz = __clzll((long long)hi);
        if (lz == 64) {
            if (lo == 0) return 0.0;
            hi = lo;
            lo = 0;
            lz = __clzll((long long)hi);
            hi <<= lz;
            lz += 64;
        } else if (lz > 0) {
            hi = hi << lz | lo >> (64 - lz);
        }
        return to_double(__umul64hi(hi, MANT), EXP - lz + x, neg);   // |F| = hi 2^(32 - lz)
    }
};
using WithH = Recombine<kNMod, kAlpha + kBeta, kHExp, kHMant, 0>;    // the product with H
using General = Recombine<kGMod, 2 * kGBits, kGExp, kGMant, 1>;      // the general products
// v[e]: elements (i + e, j), e < ROWS, where i + e < M (i a multiple of ROWS).
// The loads of kAhead moduli are in flight together: all of them where one row
// a thread leaves few threads, four with four rows, whose sums need the registers.
template <class Set, int ROWS>
__device__ __forceinline__ void recombine(int64_t i, int j, int64_t M, int64_t Mp, int mp, int nz,
                                          const uchar2 *__restrict__ R, const int *__restrict__ E,
                                          const int *__restrict__ F, z_t *v) {
    constexpr int kMods = Set::kMods, kW = Set::kWords, kW2 = (ROWS + 1) / 2;   // kW2: words of two rows
    constexpr int kAhead = ROWS == 1 ? kMods : 4;
    const int64_t step = (int64_t)mp * Mp;
    unsigned long long s[ROWS][2][kW] = {};        // [row][Re, Im][word of W]
#pragma unroll
    for (int m0 = 0; m0 < kMods; m0 += kAhead) {
        uint32_t ur[kAhead][kW2] = {}, ui[kAhead][kW2] = {};   // sums, 16 bits a row
        const uchar2 *r = R + (int64_t)j * Mp + i + (int64_t)m0 * nz * step;
#pragma unroll 1
        for (int z = 0; z < nz; z++, r += step) {
            uint32_t q[kAhead][kW2];
#pragma unroll
            for (int m = 0; m < kAhead; m++) {
                if (m0 + m >= kMods) break;
                const uchar2 *p = r + (int64_t)m * nz * step;
                if constexpr (ROWS == 4) {
                    const uint2 w = *(const uint2 *)p;
                    q[m][0] = w.x;
                    q[m][kW2 - 1] = w.y;
                } else {
                    q[m][0] = *(const uint16_t *)p;
                }
            }
#pragma unroll
            for (int m = 0; m < kAhead; m++) {
                if (m0 + m >= kMods) break;
#pragma unroll
                for (int e = 0; e < kW2; e++) {
                    ur[m][e] += q[m][e] & 0x00FF00FFu;
                    ui[m][e] += q[m][e] >> 8 & 0x00FF00FFu;
                }
            }
        }
#pragma unroll
        for (int m = 0; m < kAhead; m++) {
            if (m0 + m >= kMods) break;
#pragma unroll
            for (int k = 0; k < kW; k++) {
                const unsigned long long w = Set::word(m0 + m, k);
#pragma unroll
                for (int e = 0; e < ROWS; e++) {
                    s[e][0][k] += (ur[m][e / 2] >> (16 * (e % 2)) & 0xFFFFu) * w;
                    s[e][1][k] += (ui[m][e / 2] >> (16 * (e % 2)) & 0xFFFFu) * w;
                }
            }
        }
    }
    const int f = F[j];
#pragma unroll
    for (int e = 0; e < ROWS; e++) {
        v[e] = zmk(0.0, 0.0);
        if (i + e >= M) continue;
        const int h = E[i + e];
        if (h == INT_MIN || f == INT_MIN) continue;
        const int x = h + f - Set::kBits;
        v[e] = zmk(Set::value(s[e][0], nz, x), Set::value(s[e][1], nz, x));
    }
}

template <int ROWS>
__global__ void __launch_bounds__(128)
k_res_reduce(int64_t M, int64_t Mp, int mp, int nz, const uchar2 *__restrict__ R, const int *__restrict__ E,
             const int *__restrict__ F, GemmEpi ep, const z_t *__restrict__ Y, int64_t ldy, z_t *C,
             int64_t ldc) {
    follow();
    const int64_t i = ((int64_t)blockIdx.x * 128 + threadIdx.x) * ROWS;
    const int j = blockIdx.y;
    if (i >= M) return;
    z_t r[ROWS];
    recombine<WithH, ROWS>(i, j, M, Mp, mp, nz, R, E, F, r);
#pragma unroll
    for (int e = 0; e < ROWS; e++) {
        if (i + e >= M) break;
        z_t v = r[e];
        if (ep.mode == GEMM_CHEB) {
            v = zscale(zsub(v, zscale(Y[i + e + j * ldy], ep.c)), ep.s1);
            if (ep.Yp) v = zsub(v, zscale(ep.Yp[i + e + j * ep.ldyp], ep.s2));
        }
        C[i + e + j * ldc] = v;
    }
}

// The general products' results (RsOut).  N = 20000, 100 columns: 45 us (60 with
// the loads of two moduli in flight, 76 with conversions on the FP64 pipe too).
template <int ROWS>
__global__ void __launch_bounds__(128)
k_res_out(int64_t M, int64_t Mp, int mp, int nz, const uchar2 *__restrict__ R, const int *__restrict__ E,
          const int *__restrict__ F, RsOut o) {
    follow();
    const int64_t i = ((int64_t)blockIdx.x * 128 + threadIdx.x) * ROWS;
    const int j = blockIdx.y;
    if (i >= M) return;
    z_t r[ROWS];
    const bool lower = ROWS == 1 && o.mirror && i > j;
    recombine<General, ROWS>(lower ? j : i, lower ? (int)i : j, M, Mp, mp, nz, R, E, F, r);
    if (lower) r[0] = zconj(r[0]);
    if (ROWS == 1 && o.mirror && i == j) r[0].y = 0.0;
#pragma unroll
    for (int e = 0; e < ROWS; e++) {
        if (i + e >= M) break;
        z_t v = r[e];
        if (o.D) v = zsub(o.D[i + e + j * o.ldd], v);
        if (i + e == j) v.x += o.shift;
        if (o.adjoint) o.C[j + (i + e) * o.ldc] = zconj(v);
        else o.C[i + e + j * o.ldc] = v;
    }
}

// Whether a Gram element keeps FP64's accuracy in residues.  The operands are
// rounded to units of 2^(h - 58), 2^h >= the column's norm, so that the rms error of Re
// (or Im) G_ij is at most 2^-59.3 2^(hi + hj).  Native FP64 is accurate against
//   S = sum_k |Re a||Re b| + |Im a||Im b|   (Im: |Re a||Im b| + |Im a||Re b|)
// instead, which may lie far below the norms' product: entries far below their
// column's norm count there (a = (1, 0, ..), b = (1e-20, 1, ..)).  Where S >= 2^-4
// 2^(hi + hj) the residues' error is below 2^-55.3 S, less than one FP64 rounding of S
// (rms 2^-54.8); columns of even size have S = 0.16 .. 0.64 of it.  If any element has
// less, and not zero (whose product is exact), DEV_GRADED asks for native FP64.
// S by FP16 magnitudes relative to 2^h (entries below 2^-26 of it count as that,
// zero ones as zero) with FP32 sums, tiles of 64 x 64 columns over a part of the rows:
// straight after the norms, while A and B are in L2.  K = 20000, 140 x 40: 25 us and 6 for
// the sums, of 194 (165 without the check; native FP64: 1810).
constexpr int kWtTile = 64, kWtRows = 32;          // columns of a tile; rows staged at once
constexpr int kWtExp = 12;                         // 2^h becomes 2^12 in FP16
__device__ __forceinline__ float weight(double x, int up) {
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
    const int t = max((int)(h + (uint32_t)up), 113 << 20);     // FP32 exponent, 20 mantissa bits
    return (h | (uint32_t)__double2loint(x)) == 0 ? 0.f : __uint_as_float((uint32_t)t << 3);
}
// The same in a column of norm below 2^-1000, whose entries may all be subnormal.
__device__ __forceinline__ float weight_small(double x, int up) {
    const double a = fabs(x) * 0x1.0p1022;
    return a == 0.0 ? 0.f : fmaxf((float)ldexp(a, up / (1 << 20) - 126), 0x1.0p-14f);
}
constexpr int kUpSmall = (kWtExp + 1000 + 127 - 1023) * (1 << 20);
__device__ __forceinline__ uint32_t weights(z_t v, int up) {
    __half2 w;
    if (up <= kUpSmall) w = __floats2half2_rn(weight(v.x, up), weight(v.y, up));
    else w = __floats2half2_rn(weight_small(v.x, up), weight_small(v.y, up));
    uint32_t r;
    memcpy(&r, &w, 4);
    return r;
}
__device__ __forceinline__ void mma_16816(float *d, const uint32_t *a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// P[z][j][i]: (Re, Im) of the rows of part z.  With upper (A = B) the tiles on and
// above the diagonal alone.
__global__ void __launch_bounds__(256, 2)
k_res_weights(int64_t K, int64_t rows, int m1, int m2, const z_t *__restrict__ A, int64_t lda,
              const float2 *__restrict__ partA, const z_t *__restrict__ B, int64_t ldb,
              const float2 *__restrict__ partB, int npart, int upper, float2 *__restrict__ P) {
    __shared__ uint32_t sA[kWtTile][kWtRows + 4], sB[kWtTile][kWtRows + 4];   // (Re, Im) of a row each
    __shared__ int upA[kWtTile], upB[kWtTile];
    follow();
    if (upper && blockIdx.x > blockIdx.y) return;
    const int i0 = blockIdx.x * kWtTile, j0 = blockIdx.y * kWtTile;
    const int t = threadIdx.x, lane = t % 32, warp = t / 32;
    if (t < 2 * kWtTile) {
        const bool b = t >= kWtTile;
        const int c = t % kWtTile;
        NormAcc n;
        if (b ? j0 + c < m2 : i0 + c < m1) {
            const float2 *part = b ? partB + (int64_t)(j0 + c) * npart : partA + (int64_t)(i0 + c) * npart;
            for (int s = 0; s < npart; s++) n.add(part[s]);
        }
        const int h = n.exponent();
        (b ? upB : upA)[c] = h == INT_MIN ? 0 : (kWtExp - h + 127 - 1023) * (1 << 20);
    }
    __syncthreads();
    const int64_t kb = (int64_t)blockIdx.z * rows, ke = min(K, kb + rows);
    float acc[2][4][4] = {};                       // [Re, Im][8 columns of B][fragment]
    const int wi = warp % 4 * 16, wj = warp / 4 * 32, g = lane / 4, q = lane % 4;
    z_t va[8], vb[8];
    auto load = [&](int64_t k) {
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const int col = warp + 8 * c;
            va[c] = (k < ke && i0 + col < m1) ? A[k + (i0 + col) * lda] : zmk(0.0, 0.0);
            vb[c] = (k < ke && j0 + col < m2) ? B[k + (j0 + col) * ldb] : zmk(0.0, 0.0);
        }
    };
    load(kb + lane);
    for (int64_t k0 = kb; k0 < ke; k0 += kWtRows) {
        if (k0 > kb) __syncthreads();              // the step before has been read
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const int col = warp + 8 * c;
            sA[col][lane] = i0 + col < m1 ? weights(va[c], upA[col]) : 0;
            sB[col][lane] = j0 + col < m2 ? weights(vb[c], upB[col]) : 0;
        }
        __syncthreads();
        load(k0 + kWtRows + lane);                 // under way during the products
#pragma unroll
        for (int s = 0; s < kWtRows; s += 8) {
            const uint32_t a[4] = {sA[wi + g][s + q], sA[wi + g + 8][s + q], sA[wi + g][s + q + 4], sA[wi + g + 8][s + q + 4]};
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const uint32_t b0 = sB[wj + 8 * n + g][s + q], b1 = sB[wj + 8 * n + g][s + q + 4];
                mma_16816(acc[0][n], a, b0, b1);
                mma_16816(acc[1][n], a, __byte_perm(b0, 0, 0x1032), __byte_perm(b1, 0, 0x1032));
            }
        }
    }
    float2 *Pz = P + (int64_t)blockIdx.z * m1 * m2;
#pragma unroll
    for (int n = 0; n < 4; n++)
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int i = i0 + wi + g + (e >= 2 ? 8 : 0), j = j0 + wj + 8 * n + 2 * q + (e & 1);
            if (i < m1 && j < m2) Pz[(int64_t)j * m1 + i] = make_float2(acc[0][n][e], acc[1][n][e]);
        }
}
// 32 elements a block, their parts over 8 warps.
__global__ void __launch_bounds__(256)
k_res_weigh(int m1, int m2, int nz, const float2 *__restrict__ P, int upper, ChaseScalars *sc) {
    __shared__ float2 part[8][32];
    follow();
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int64_t n = (int64_t)m1 * m2, e = (int64_t)blockIdx.x * 32 + lane;
    const int i = (int)(e % m1), j = (int)(e / m1);
    const bool in = e < n && !(upper && i > j);
    float2 s = make_float2(0.f, 0.f);
    if (in) {
#pragma unroll 4
        for (int z = warp; z < nz; z += 8) {
            const float2 p = P[(int64_t)z * n + e];
            s.x += p.x;
            s.y += p.y;
        }
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || !in) return;
    for (int w = 1; w < 8; w++) {
        s.x += part[w][lane].x;
        s.y += part[w][lane].y;
    }
    constexpr float least = (float)(1 << (2 * kWtExp - 4));
    if (upper && i == j) s.y = 0.f;                // the diagonal is real
    if ((s.x > 0.f && s.x < least) || (s.y > 0.f && s.y < least)) set_error(sc, DEV_GRADED, j);
}

// 3-D FP16 tensor [tiles][rows][64], box 64 x box_rows x box_tiles, 128-byte swizzle
bool make_map(CUtensorMap *m, void *base, uint64_t rows, uint64_t tiles, uint32_t box_rows, uint32_t box_tiles) {
    const TensorMapEncode enc = tensor_map_encode();
    if (!enc) return false;
    cuuint64_t dims[3] = {64, rows, tiles};
    cuuint64_t strides[2] = {64 * 2, rows * 64 * 2};
    cuuint32_t box[3] = {64, box_rows, box_tiles};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, base, dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Column tiles of an n-column product: as few as hold n, of equal width
void column_tiles(int n, int *tx, int *w) {
    *tx = (n + kMaxW - 1) / kMaxW;
    *w = ((n + *tx - 1) / *tx + 15) / 16 * 16;
}

// Parts of B's residues for a tile of w columns: Re and Im, and with Gauss their sum
int b_parts(int w) { return w > kGaussW ? 3 : 2; }

// Chunks per K split.  Modelled time, in cycles, of the busiest SM: a chunk
// takes 6 or 8 w cycles of MMA, at least about 700 (its share of HBM) or 260 (its
// conversion) when the matrix is in L2; a unit costs about 2000 more (its first
// copies and its last drain) and each split about 52 bytes per output.
int choose_chunks(int64_t Mp, int nch, int mp, int tx, int w, int nmod, size_t r_bytes, int sms) {
    const double mat = 2.0 * nmod * Mp * nch * kChunk;
    const double per_chunk = std::max((w > kGaussW ? 6.0 : 8.0) * w, mat > 1.0e8 ? 700.0 : 300.0);
    const int64_t tiles = Mp / kRows * tx * nmod;
    int best = 0;
    double best_t = 1e300;
    for (int cs = 1; cs <= kMaxUnitChunks; cs = cs < 8 ? cs * 2 : cs + 8) {
        const int nz = (nch + cs - 1) / cs;
        if (nz > 250) continue;                    // 16-bit sums of the splits' bytes
        if ((size_t)nmod * nz * mp * Mp * sizeof(uchar2) > r_bytes) continue;
        const int64_t per = (tiles * nz + sms - 1) / sms;
        const double t = (double)per * (std::min(cs, nch) * per_chunk + 2000.0) +
                         4.0 * nmod * nz * mp * Mp / (5e12 / 1.9e9);
        if (t < best_t) {
            best_t = t;
            best = cs;
        }
    }
    return best;
}

int norm_segment(int64_t N) { return N <= 1024 ? 8 : N < 4096 ? 32 : 256; }
constexpr int64_t kShortColumn = 4096;

}  // namespace

namespace {
size_t a_bytes_of(int64_t M, int64_t K, int nmod) {
    const int64_t Mp = (M + kRows - 1) / kRows * kRows, Kp = (K + kChunk - 1) / kChunk * kChunk;
    return (size_t)nmod * 2 * Mp * Kp;
}
size_t b_bytes_of(int64_t K, int n, int nmod) {
    const int64_t Kp = (K + kChunk - 1) / kChunk * kChunk;
    return (size_t)nmod * 3 * Kp * (n + 64) * 2;
}
}  // namespace

size_t residue_a_bytes(int64_t M, int64_t K) { return a_bytes_of(M, K, kNMod); }

size_t residue_b_bytes(int64_t K, int n) { return b_bytes_of(K, n, kNMod); }

size_t residue_r_bytes(int64_t M, int64_t K, int n) {
    const int64_t Mp = (M + kRows - 1) / kRows * kRows, nch = (K + kChunk - 1) / kChunk;
    // splits: as many as the longest units need, and some more to fill the SMs
    const int64_t nz = std::max<int64_t>((nch + kMaxUnitChunks - 1) / kMaxUnitChunks, std::min<int64_t>(nch, nch < 128 ? 8 : 3));
    return (size_t)kNMod * nz * (n + 64) * Mp * sizeof(uchar2);
}

size_t residue_work_bytes(int64_t N) {
    const int64_t s = norm_segment(N);
    return (size_t)((N + s - 1) / s) * N * sizeof(float2);
}

size_t residue_panel_bytes(int64_t N) { return (size_t)N * 256 * sizeof(z_t); }

cudaError_t residue_prepare(int64_t N, const z_t *H, int64_t ldh, OzakiH *oh, void *work, ChaseScalars *sc, int sms,
                            cudaStream_t st) {
    const int64_t Np = ozaki_padded(N), T = Np / kRows, nch = (N + kChunk - 1) / kChunk;
    oh->N = N;
    oh->Np = Np;
    oh->tri = false;
    const int seg = norm_segment(N), nseg = (int)((N + seg - 1) / seg);
    const unsigned rb = (unsigned)((N + 127) / 128);
    if (seg < 256 && nseg <= kSmallSegs) {
        launch_next(k_res_rowexp<8, 64, kSmallSegs>, dim3((unsigned)(Np / 8)), dim3(512), 0, st, N, Np, N, H, ldh, seg,
                    nseg, oh->E, sc);
        bse_count_launches(1);
    } else {
        k_res_rownorm<<<dim3(rb, (unsigned)nseg), 128, 0, st>>>(N, N, H, ldh, seg, 0, (float2 *)work);
        k_res_rowscale<<<(unsigned)T, 128, 0, st>>>(N, Np, nseg, (const float2 *)work, oh->E, sc);
        bse_count_launches(2);
    }
    if (nch * 4 * T < 4 * sms)                     // too few blocks for four on every SM (N = 256: 9.2 us, 6.5 here)
        launch_next(k_res_slice_a<4>, dim3((unsigned)(nch * 16), (unsigned)T), dim3(128), 0, st, N, N, H, ldh, (int64_t)0, T,
                    nch, oh->E, kNMod, kAlpha, (uint8_t *)oh->A);
    else
        launch_next(k_res_slice_a<16>, dim3((unsigned)(nch * 4), (unsigned)T), dim3(128), 0, st, N, N, H, ldh, (int64_t)0, T,
                    nch, oh->E, kNMod, kAlpha, (uint8_t *)oh->A);
    bse_count_launches(1);
    return cudaGetLastError();
}

cudaError_t residue_prepare_bse(int Nk, int Nv, int Nc, const BseModel &md, const double *dE, const z_t *u,
                                const z_t *a, const double *Kt, OzakiH *oh, void *work, void *panel,
                                ChaseScalars *sc, cudaStream_t st) {
    const int64_t N = (int64_t)Nk * Nv * Nc, Np = ozaki_padded(N), T = Np / kRows, nch = (N + kChunk - 1) / kChunk;
    oh->N = N;
    oh->Np = Np;
    oh->tri = false;
    const int dyn = 2 * kPT * std::max(md.rank_x, 1) * (int)sizeof(z_t);
    static std::once_flag once[kMaxDevices];
    static cudaError_t attr[kMaxDevices];
    const cudaError_t ae = smem_attr_once(once, attr, (const void *)k_res_panel, 2 * kPT * 64 * (int)sizeof(z_t));
    if (ae != cudaSuccess) return ae;
    const int seg = norm_segment(N), nseg = (int)((N + seg - 1) / seg);
    const unsigned rb = (unsigned)((N + 127) / 128);
    z_t *Hp = (z_t *)panel;
    for (int pass = 0; pass < 2; pass++) {
        for (int64_t j0 = 0; j0 < N; j0 += 256) {
            const int cols = (int)std::min<int64_t>(256, N - j0);
            k_res_panel<<<dim3((unsigned)((N + kPT - 1) / kPT), (unsigned)((cols + kPT - 1) / kPT)),
                          dim3(kPT, 8), dyn, st>>>(Nk, Nv * Nc, (int)N, (int)j0, cols, md, dE, u, a, Kt, Hp);
            if (pass == 0)
                k_res_rownorm<<<dim3(rb, (unsigned)((cols + seg - 1) / seg)), 128, 0, st>>>(
                    N, cols, Hp, N, seg, j0 / seg, (float2 *)work);
            else
                k_res_slice_a<16><<<dim3((unsigned)((cols + kChunk - 1) / kChunk * 4), (unsigned)T), 128, 0, st>>>(
                    N, N, Hp, N, j0, T, nch, oh->E, kNMod, kAlpha, (uint8_t *)oh->A);
            bse_count_launches(2);
        }
        if (pass == 0) {
            k_res_rowscale<<<(unsigned)T, 128, 0, st>>>(N, Np, nseg, (const float2 *)work, oh->E, sc);
            bse_count_launches(1);
        }
    }
    return cudaGetLastError();
}

double residue_flops(int64_t M, int64_t K, int n) {
    int tx, w;
    column_tiles(n, &tx, &w);
    return (w > kGaussW ? 6.0 : 8.0) * kNMod * (double)M * (double)K * n;
}

namespace {
template <class Cfg>
cudaError_t launch_cfg(RsBatch &b, int sms, cudaStream_t st) {
    b.slots = std::min((kTmemCols - 3 * b.stride) / Cfg::kCols, kMaxSlots);
    static std::once_flag once[kMaxDevices];
    static cudaError_t attr[kMaxDevices];
    const cudaError_t ae = smem_attr_once(once, attr, (const void *)k_res_zgemm<Cfg>, Cfg::kSmem);
    if (ae != cudaSuccess) return ae;
    launch_next(k_res_zgemm<Cfg>, dim3((unsigned)std::min(b.units, sms)), dim3(Cfg::kThreads), Cfg::kSmem, st, b);
    bse_count_launches(1);
    return cudaGetLastError();
}
}  // namespace

bool rs_gauss(const RsJob &j) { return j.w > kGaussW; }

cudaError_t residue_launch(RsBatch &b, int sms, cudaStream_t st) {
    b.stride = 16;
    for (int j = 0; j < b.njobs; j++) b.stride = std::max(b.stride, b.job[j].w);
    if (b.stride <= RsNarrow::kW) return launch_cfg<RsNarrow>(b, sms, st);
    if (b.stride <= RsMid::kW) return launch_cfg<RsMid>(b, sms, st);
    if (b.stride <= kGaussW) return launch_cfg<RsWide>(b, sms, st);
    return launch_cfg<RsGauss>(b, sms, st);
}

namespace {
// A launch of one product: the residues of A (Mp rows) and of B (tx tiles of w columns)
bool single_job(RsBatch *b, const void *A, void *B, int64_t Mp, int nch, int tx, int w, int nmod, void *R,
                size_t r_bytes, ChaseScalars *sc, uint64_t wait_ns, int sms) {
    memset(b, 0, sizeof *b);
    RsJob &j = b->job[0];
    const int mp = tx * w;
    if (!make_map(&j.tmB, B, (uint64_t)mp, (uint64_t)nmod * b_parts(w) * nch, (uint32_t)w, w > kGaussW ? 1 : 2))
        return false;
    j.A = (const uint8_t *)A;
    j.R = (uchar2 *)R;
    j.sc = sc;
    j.wait_ns = wait_ns;
    j.Mp = Mp;
    j.w = w;
    j.mp = mp;
    j.nch = nch;
    j.cs = choose_chunks(Mp, nch, mp, tx, w, nmod, r_bytes, sms);
    if (j.cs < 1) return false;
    j.tx = tx;
    j.ty = (int)(Mp / kRows);
    j.tz = (nch + j.cs - 1) / j.cs;
    j.nmod = nmod;
    b->njobs = 1;
    b->units = rs_units(j);
    return true;
}
}  // namespace

cudaError_t residue_zgemm(const OzakiH &oh, int n, const z_t *Y, int64_t ldy, z_t *C, int64_t ldc,
                          const GemmEpi &ep, void *B, size_t b_bytes, int *F, float2 *part, void *R,
                          size_t r_bytes, ChaseScalars *sc, int sms, cudaStream_t st, cudaEvent_t ev0,
                          cudaEvent_t ev1, OzBatcher *batcher) {
    if (n <= 0) return cudaSuccess;
    const int64_t N = oh.N, nch = (N + kChunk - 1) / kChunk, Kp = nch * kChunk;
    int tx, w;
    column_tiles(n, &tx, &w);
    const int mp = tx * w;
    if ((size_t)kNMod * 3 * Kp * mp * 2 > b_bytes) return cudaErrorInvalidValue;
    // a short column's norm is taken by each block that slices a part of it (N =
    // 2000, 75 columns: 11.6 us against 5.9 for the norms and 8.8)
    const int npart = N <= kShortColumn ? 0 : (int)std::min<int64_t>((N + 1023) / 1024, 32);
    if (npart > 0) {
        launch_next(k_res_colnorm, dim3((unsigned)npart, (unsigned)n), dim3(256), 0, st, N, Y, ldy, part, sc);
        bse_count_launches(1);
    }
    const unsigned bx = (unsigned)((Kp + 1023) / 1024);
    // split the moduli over blocks while that leaves SMs idle otherwise
    const unsigned bz = (unsigned)std::max<int64_t>(1, std::min<int64_t>(kNMod, 4 * sms / ((int64_t)bx * mp)));
    launch_next(k_res_slice_b, dim3(bx, (unsigned)mp, bz), dim3(128), 0, st, N, Kp, n, mp, Y, ldy, npart, part, F, kNMod,
                kBeta, b_parts(w), (uint16_t *)B, sc);
    bse_count_launches(1);
    RsBatch b;
    RsJob &j = b.job[0];
    if (!single_job(&b, oh.A, B, oh.Np, (int)nch, tx, w, kNMod, R, r_bytes, sc, oh.wait_ns, sms))
        return cudaErrorInvalidValue;
    cudaError_t e;
    if (batcher) {
        e = ozb_run_residue(batcher, j, st);
    } else {
        if (ev0) cudaEventRecord(ev0, st);
        e = residue_launch(b, sms, st);
        if (ev1) cudaEventRecord(ev1, st);
    }
    if (e != cudaSuccess) return e;
    if (N * n < 400000)                            // too few threads at four rows each
        launch_next(k_res_reduce<1>, dim3((unsigned)((N + 127) / 128), (unsigned)n), dim3(128), 0, st, N, oh.Np, mp, j.tz,
                    j.R, oh.E, F, ep, Y, ldy, C, ldc);
    else
        launch_next(k_res_reduce<4>, dim3((unsigned)((N + 511) / 512), (unsigned)n), dim3(128), 0, st, N, oh.Np, mp, j.tz,
                    j.R, oh.E, F, ep, Y, ldy, C, ldc);
    bse_count_launches(1);
    return cudaGetLastError();
}

// ------------------------------------------------------------ general products
// A^H B and A B of the QR and Gram entries, for tall A and B.  In native FP64
// (1.2 TFLOP/s on this part) they were bound by its issue: Gram K = 20000,
// 140 x 40: 1805 us, here 197 (55 left residues, 23 right, 21 norms, 31 their weights'
// check, 39 product, 8 result); QR N = 20000, 100 columns after 40: 21.8 ms, here 2.8.
size_t residue_left_bytes(int64_t M, int64_t K) { return a_bytes_of(M, K, kGMod); }
size_t residue_right_bytes(int64_t K, int n) { return b_bytes_of(K, n, kGMod); }
size_t residue_out_bytes(int64_t M, int64_t K, int n) {
    const int64_t Mp = (M + kRows - 1) / kRows * kRows, nch = (K + kChunk - 1) / kChunk;
    // splits of a long sum: enough to fill the SMs from one row tile
    const int64_t nz = std::max<int64_t>((nch + kMaxUnitChunks - 1) / kMaxUnitChunks, std::min<int64_t>(nch, Mp <= 512 ? 24 : 4));
    return (size_t)kGMod * nz * (n + 64) * Mp * sizeof(uchar2);
}

namespace {
int col_parts(int64_t K) { return (int)std::min<int64_t>((K + 1023) / 1024, kRsColParts); }

void col_norms(int64_t K, int64_t n, const z_t *A, int64_t lda, float2 *part, ChaseScalars *sc, cudaStream_t st) {
    launch_next(k_res_colnorm, dim3((unsigned)col_parts(K), (unsigned)n), dim3(256), 0, st, K, A, lda, part, sc);
    bse_count_launches(1);
}
}  // namespace

cudaError_t residue_left(int64_t M, int64_t K, const z_t *A, int64_t lda, bool ah, const RsSide &s, ChaseScalars *sc,
                         cudaStream_t st, bool normed) {
    const int64_t T = (M + kRows - 1) / kRows, nch = (K + kChunk - 1) / kChunk;
    if (M < 1 || K < 1 || residue_left_bytes(M, K) > s.bytes || (!ah && K > kMaxTallCols)) return cudaErrorInvalidValue;
    if (ah) {
        if (!normed) col_norms(K, M, A, lda, s.part, sc, st);
        launch_next(k_res_slice_ah, dim3((unsigned)nch, (unsigned)((M + 31) / 32)), dim3(128), 0, st, M, K, A, lda, T, nch,
                    col_parts(K), s.part, s.e, kGMod, kGBits, (uint8_t *)s.p);
    } else {
        launch_next(k_res_rowexp<32, 8, kTallSegs>, dim3((unsigned)(T * kRows / 32)), dim3(256), 0, st, M, T * kRows, K, A,
                    lda, 32, (int)((K + 31) / 32), s.e, sc);
        launch_next(k_res_slice_a<16>, dim3((unsigned)(nch * 4), (unsigned)T), dim3(128), 0, st, M, K, A, lda, (int64_t)0, T,
                    nch, s.e, kGMod, kGBits, (uint8_t *)s.p);
        bse_count_launches(1);
    }
    bse_count_launches(1);
    return cudaGetLastError();
}

cudaError_t residue_right(int64_t K, int n, const z_t *B, int64_t ldb, const float2 *norms, const RsSide &s,
                          ChaseScalars *sc, int sms, cudaStream_t st) {
    if (n < 1 || K < 1 || residue_right_bytes(K, n) > s.bytes) return cudaErrorInvalidValue;
    const int64_t Kp = (K + kChunk - 1) / kChunk * kChunk;
    int tx, w;
    column_tiles(n, &tx, &w);
    const int mp = tx * w;
    int npart = 0;
    if (norms || K > kShortColumn) {
        if (!norms) col_norms(K, n, B, ldb, s.part, sc, st);
        npart = col_parts(K);
    }
    const unsigned bx = (unsigned)((Kp + 1023) / 1024);
    const unsigned bz = (unsigned)std::max<int64_t>(1, std::min<int64_t>(kGMod, 4 * sms / ((int64_t)bx * mp)));
    launch_next(k_res_slice_b, dim3(bx, (unsigned)mp, bz), dim3(128), 0, st, K, Kp, n, mp, B, ldb, npart,
                norms ? norms : s.part, s.e, kGMod, kGBits, b_parts(w), (uint16_t *)s.p, sc);
    bse_count_launches(1);
    return cudaGetLastError();
}

cudaError_t residue_product(int64_t M, int n, int64_t K, const RsSide &A, const RsSide &B, const RsOut &out, void *R,
                            size_t r_bytes, uint64_t wait_ns, ChaseScalars *sc, int sms, cudaStream_t st) {
    if (out.mirror && (M != n || out.adjoint || out.D)) return cudaErrorInvalidValue;
    const int64_t Mp = (M + kRows - 1) / kRows * kRows, nch = (K + kChunk - 1) / kChunk;
    int tx, w;
    column_tiles(n, &tx, &w);
    RsBatch b;
    if (!single_job(&b, A.p, B.p, Mp, (int)nch, tx, w, kGMod, R, r_bytes, sc, wait_ns, sms)) return cudaErrorInvalidValue;
    const RsJob &j = b.job[0];
    const cudaError_t e = residue_launch(b, sms, st);
    if (e != cudaSuccess) return e;
    if (M * n < 400000 || out.mirror)
        launch_next(k_res_out<1>, dim3((unsigned)((M + 127) / 128), (unsigned)n), dim3(128), 0, st, M, Mp, j.mp, j.tz, j.R,
                    A.e, B.e, out);
    else
        launch_next(k_res_out<4>, dim3((unsigned)((M + 511) / 512), (unsigned)n), dim3(128), 0, st, M, Mp, j.mp, j.tz, j.R,
                    A.e, B.e, out);
    bse_count_launches(1);
    return cudaGetLastError();
}

cudaError_t residue_norms(int64_t K, int n, const z_t *A, int64_t lda, float2 *part, ChaseScalars *sc, cudaStream_t st) {
    if (n < 1 || K < 1) return cudaErrorInvalidValue;
    col_norms(K, n, A, lda, part, sc, st);
    return cudaGetLastError();
}

cudaError_t residue_weigh(int64_t K, int m1, int m2, const z_t *A, int64_t lda, const float2 *normsA, const z_t *B,
                          int64_t ldb, const float2 *normsB, bool same, void *work, size_t bytes, ChaseScalars *sc,
                          int sms, cudaStream_t st) {
    const int64_t tx = (m1 + kWtTile - 1) / kWtTile, ty = (m2 + kWtTile - 1) / kWtTile, n = (int64_t)m1 * m2;
    // parts of 128 rows at least, and as many as fill the SMs and `work` holds
    int64_t nz = std::min<int64_t>((K + 127) / 128, std::max<int64_t>(1, 2 * sms / (tx * ty)));
    nz = std::min<int64_t>(nz, (int64_t)(bytes / (n * sizeof(float2))));
    if (nz < 1) return cudaErrorInvalidValue;
    const int64_t rows = ((K + nz - 1) / nz + kWtRows - 1) / kWtRows * kWtRows;
    nz = (K + rows - 1) / rows;
    launch_next(k_res_weights, dim3((unsigned)tx, (unsigned)ty, (unsigned)nz), dim3(256), 0, st, K, rows, m1, m2, A, lda,
                normsA, B, ldb, normsB, col_parts(K), same ? 1 : 0, (float2 *)work);
    launch_next(k_res_weigh, dim3((unsigned)((n + 31) / 32)), dim3(256), 0, st, m1, m2, (int)nz, (const float2 *)work,
                same ? 1 : 0, sc);
    bse_count_launches(2);
    return cudaGetLastError();
}
