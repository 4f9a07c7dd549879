// Hybrid key switching on rings of 2^10 points and more, after the lift (ntt.cu): the second half of every digit's forward
// transform, the product with the key and the sum over rotations in one kernel; the second half of the ModDown transforms and
// the final combination in another.  Neither the transformed digits nor the transformed ModDown polynomials travel to memory.
//
// Positions.  A polynomial is stored in chunks of 256 words with their low nibbles swapped (see galois_src): word m = 16 b + a of
// a chunk holds logical position 16 a + b.  Sixteen lanes (a half-warp) transform one chunk of one polynomial in two register
// rounds; lane j holds logical positions j + 16 e in the first forward round and 16 j + e in the second.  In shared memory logical
// position 16 a + b is kept at word 16 a + (b ^ a), which both rounds and the word-by-word passes reach without bank conflicts
// (swz).  An automorphism maps every chunk of 256 positions onto one chunk, so a CTA that owns a chunk of the result reads
// one chunk of every source and permutes inside it.
#include <algorithm>

#include "internal.h"
#include "debugcheck.cuh"
#include "nttcore.cuh"

namespace {

__device__ __forceinline__ int swz(int m) { return ((m & 15) << 4) | ((m >> 4) ^ (m & 15)); }

// The words 16 e + j of a chunk (logical positions 16 j + e) under an automorphism: their sources share the chunk and the low nibble
// of the word; the high nibble, bit-reversed, advances by k times the bit-reversed e.
struct LaneSource {
    int base;  // first word of the source chunk + the low nibble
    unsigned t0, k;
    __device__ __forceinline__ static int brev4(unsigned v) { return (int)((0xF7B3D591E6A2C480ULL >> (4 * v)) & 15); }
    __device__ __forceinline__ LaneSource(int first, unsigned k_, int logN) : k(k_) {
        const int s = galois_src(first, k_, logN, 1);
        base = s & ~0xF0;
        t0 = brev4((s >> 4) & 15);
    }
    __device__ __forceinline__ int high(int e) const { return brev4((t0 + brev4(e) * k) & 15); }
    __device__ __forceinline__ int word(int e) const { return base + 16 * high(e); }
};

// table entries of a chunk's second pass (cbase = 2^a + chunk number) in the order of the two rounds: entries 0..14 for the first
// round (broadcast to the lanes of a chunk), entry 16 (r + 1) + j, r = 2^u - 1 + il, for stage u of the second
template <class TW>
__device__ __forceinline__ void stage_twiddles(TW* __restrict__ tc, const TW* __restrict__ tw, unsigned cbase) {
#pragma unroll 4
    for (int e = threadIdx.x; e < 256; e += blockDim.x) {
        const int r = e < 16 ? e : (e >> 4) - 1, u = 31 - __clz(r + 1), il = r + 1 - (1 << u);
        const unsigned idx = e < 16 ? (cbase << u) + il : (cbase << (4 + u)) + ((e & 15) << u) + il;
        if (r < 15) tc[e] = tw[idx];
    }
}

// 16-byte asynchronous copies of the 2 L key chunks (256 words each, KN words apart) of a modulus into shared memory
__device__ __forceinline__ void stage_keys(u64* __restrict__ ks, const u64* __restrict__ key, long long KN, int L) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(ks);
    for (int v = threadIdx.x; v < 2 * L * 128; v += blockDim.x) {
        const u64* src = key + (long long)(v >> 7) * KN + (v & 127) * 2;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + v * 16), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// the eight stages of a chunk: x[e] enters as word j + 16 e (pass-A format) and leaves as logical position 16 j + e, unreduced
// (below 8q)
__device__ __forceinline__ void chunk_forward(const ArithF64& ar, double (&x)[16], const double2* tc, u64* sb, int j, unsigned hmask) {
    fwd_round_f<4, ArithF64, 4>(ar, x, [=](int st, int il) { return tc[(1 << st) - 1 + il]; });
#pragma unroll
    for (int e = 0; e < 16; e++) sb[16 * e + (j ^ e)] = ar.to_exch(x[e]);
    __syncwarp(hmask);
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = ar.from_mid(sb[16 * j + (e ^ j)]);
    fwd_round_f<4, ArithF64, 1>(ar, x, [=](int u, int il) { return tc[(((1 << u) + il) << 4) + j]; });
}
// the same in place for the integer classes, rolled (see fwd_round4_smem): x[e] enters at the word of position j + 16 e; canonical
// residues at the words of the swizzled layout
template <class AR>
__device__ __forceinline__ void chunk_forward_int(const AR& ar, const ulonglong2* tc, u64* sb, int j, unsigned hmask) {
    fwd_round4_staged(ar, [=](int e) { return sb + 16 * e + (j ^ e); }, tc, 1, 0);
    __syncwarp(hmask);
    const auto second = [=](int e) { return sb + 16 * j + (e ^ j); };
    fwd_round4_staged(ar, second, tc + 16, 16, j);
#pragma unroll 2
    for (int e = 0; e < 16; e++) *second(e) = ar.to_canonical(*second(e));
}

// the inverse table's entries of a chunk (cbase = 2^a + chunk number) in the order of the two inverse rounds: entry 16 (r + 1) + j,
// r = 16 - (16 >> st) + il, for stage st of the first, entries 0..14 (r) for the second
template <class TW>
__device__ __forceinline__ void stage_inverse_twiddles(TW* __restrict__ tc, const TW* __restrict__ tw, unsigned cbase) {
#pragma unroll 4
    for (int e = threadIdx.x; e < 256; e += blockDim.x) {
        const int r = e < 16 ? e : (e >> 4) - 1, s = r < 8 ? 0 : r < 12 ? 1 : r < 14 ? 2 : 3, il = r - (16 - (16 >> s));
        const unsigned idx = ((e < 16 ? cbase : (cbase << 4) + (e & 15)) << (3 - s)) + il;
        if (r < 15) tc[e] = tw[idx];
    }
}

// inverse pass B' of a chunk (cbase = 2^a + chunk number) by sixteen lanes, lane j holding its logical positions 16 j + e at the words
// sv[16 j + (e ^ j)] (balanced binary64 integers, or residues in [0, 2q)); the chunk in the private format at o.  STAGED: tw is what
// stage_inverse_twiddles left, otherwise the table of the modulus
template <bool STAGED>
__device__ __forceinline__ void chunk_inverse(const ArithF64& ar, const double2* __restrict__ tw, unsigned cbase, u64* sv, u64* o, int j, unsigned hmask) {
    double x[16];
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = ar.from_mid(sv[16 * j + (e ^ j)]);
    if (STAGED) inv_round_f<4>(ar, x, [=](int st, int il) { return tw[((16 - (16 >> st) + il + 1) << 4) + j]; });
    else inv_round<4>(ar, x, tw, (cbase << 4) + j);
#pragma unroll
    for (int e = 0; e < 16; e++) sv[16 * j + (e ^ j)] = ar.to_mid(x[e]);
    __syncwarp(hmask);
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = ar.from_mid(sv[16 * e + (j ^ e)]);
    if (STAGED) inv_round_f<4>(ar, x, [=](int st, int il) { return tw[16 - (16 >> st) + il]; });
    else inv_round<4>(ar, x, tw, cbase);
#pragma unroll
    for (int e = 0; e < 16; e++) o[j + 16 * e] = ar.to_mid(x[e]);
}
template <bool STAGED>
__device__ __forceinline__ void chunk_inverse(const ArithInt<false>& ar, const ulonglong2* __restrict__ tw, unsigned cbase, u64* sv, u64* o, int j, unsigned hmask) {
    const auto first = [=](int e) { return sv + 16 * j + (e ^ j); };
    const auto second = [=](int e) { return sv + 16 * e + (j ^ e); };
    if (STAGED) inv_round4_staged(ar, first, tw + 16, 16, j);
    else inv_round4_smem(ar, first, tw, (cbase << 4) + j);
    __syncwarp(hmask);
    if (STAGED) inv_round4_staged(ar, second, tw, 1, 0);
    else inv_round4_smem(ar, second, tw, cbase);
#pragma unroll 8
    for (int e = 0; e < 16; e++) o[j + 16 * e] = *second(e);
}

struct ApplyArgs {
    const u64* digits;  // pass-A output of digit (z, item, j) for modulus i: ((z * items + item) * L + j) * n_tgt + target of i
    int n_tgt;          // targets per digit: L + 1; or one less, a digit's own modulus being left out and read from `own`; with
                        // auxiliary primes none for the special prime either
    int nx;             // 1, or the number of auxiliary primes that stand for the special prime
    u64 aux4;           // their limbs in 4-bit fields, behind them the other limbs
    long long aux_key;  // and the offset of their words in a key
    const u64* own;     // the polynomials being switched, transform domain: own + item * own_it + z * own_z + j * N (or null)
    long long own_it, own_z;
    const u64* const* keytab;
    const unsigned* galois;
    int rot0, rot_zinc, nz;  // rotation of z
    long long items;
    u64* u;  // [item][2][L+nx][N]: limbs below L canonical (below 2^50: balanced binary64 integers), the special prime's (or the
             // auxiliary primes') after inverse pass B' (private format)
    int N, logN, L;
    const void *tw_fwd_f64, *tw_fwd_int, *tw_inv_f64, *tw_inv_int;
    const LimbConst* lt;
};

// u[item][c][i] = sum over z of phi_z( sum_j digit(z, item, j) * key_z[j][c] )  modulo i, for chunk blockIdx.x of the result, a modulus
// per blockIdx.y (the special prime or the auxiliary ones, which have the longest chain, first) and IB items.  A half-warp transforms one digit's
// chunk; then every thread multiplies positions of all items with key words it loads once.
//
// Bound: issue slots and FP64 pipe together (ncu, two items x three z at N = 2^16, L = 4: FP64 27 %, issue 51 %, 96 registers and 20
// warps per SM; 80 registers and 24 warps were 2 to 3 % slower).  The table entries and key words of a chunk are staged in shared
// memory (the keys asynchronously, under the transform), which took the single-item launch from 91 to 51 us: read from global
// memory they sat in the chain.  The sums are reduced on the FP64 pipe: the 128-bit integer reduction was as long as the products.
// Against pass B, key product and permuted sum as kernels of their own (seven blocks, three giant steps, N = 2^16, L = 4):
// 513 -> 390 us with the finish kernel below, and four of twenty digit transforms less in the lift.
//
// SHARE (with auxiliary primes): the CTA of an auxiliary prime takes the products with the key modulo that prime as well, instead of a
// CTA of their own that transforms the same digits again; both key sets and sums then wait in shared memory.  At four items per CTA that
// is 104 KiB, two CTAs per SM as without: 31 blocks of three rotations 1163 -> 840 us.  At one and two items it leaves three
// CTAs in place of five and lost (95 -> 108 us for two).
template <int IB, int T, bool SHARE>
__global__ void __launch_bounds__(T, 640 / T) k_ks_apply(ApplyArgs A) {
    extern __shared__ __align__(16) u64 sm[];
    const int L = A.L, N = A.N, t = blockIdx.x, y = blockIdx.y;
    const bool last = y < A.nx, aux = last && A.nx > 1;
    const int i = SHARE || aux ? (int)(A.aux4 >> (4 * y)) & 15 : last ? L : y - A.nx;
    const int sets = aux ? 2 : 1;  // SHARE: key sets, 0 the modulus' own, 1 the auxiliary one
    const long long UN = (long long)(L + A.nx) * N;
    // (the inverse table is staged where enough threads share that: a launch of CTAs of 64 threads was 7 % slower with it, one of 256
    // 10 % faster)
    constexpr bool INV = T >= 256;
    double2* tc = (double2*)sm;                  // [256] forward, INV: [256] inverse
    u64* ks = sm + (INV ? 1024 : 512);           // [L][2][256] key words of a set, those of the second behind the sums
    u64* buf = ks + (size_t)L * 512;             // [IB * L][256] digits
    u64* acc = buf + (size_t)IB * L * 256;       // [IB][2][256] sums of a set
    // words from the first set's buffers to the second's
    const int ks2 = SHARE ? L * 512 + IB * (L * 256 + 512) : 0, acc2 = SHARE ? IB * 512 + L * 512 : 0;
    const long long it0 = (long long)blockIdx.z * IB;
    const int nit = A.items - it0 < IB ? (int)(A.items - it0) : IB;
    const int hw = threadIdx.x >> 4, j = threadIdx.x & 15;
    const unsigned hmask = 0xFFFFu << (threadIdx.x & 16);
    const LimbConst* lc = A.lt + i;
    const u64 q = lc->q;
    const bool f64 = q < (1ULL << 50);
    const unsigned m0 = (unsigned)(N >> 8);
    const int it = hw / L, dj = hw - it * L;
    const bool valid = it < nit, own = A.own && dj == i;
    u64* sb = buf + hw * 256;
    const ArithF64 ar(lc);
    const double2 c51 = make_double2(lc->c51_bal, lc->c51_q);
    int staged = -1;
    for (int z = 0; z < A.nz; z++) {
        const unsigned k = A.galois[A.rot0 + z * A.rot_zinc];
        const int sc = k == 1u ? t : galois_src(t << 8, k, A.logN, 1) >> 8;
        const u64* p = own ? A.own + (it0 + it) * A.own_it + z * A.own_z + (long long)i * N
                           : A.digits + (((z * A.items + it0 + it) * L + dj) * A.n_tgt + (!A.own || i < dj ? i : i - 1)) * N;
        p += (sc << 8);
        if (z) __syncthreads();  // the products of the previous rotation have been taken
        const u64* key = A.keytab[A.rot0 + z * A.rot_zinc] + (sc << 8);
        if (SHARE || !aux) stage_keys(ks, key + (long long)i * N, (long long)(L + 1) * N, L);
        if (aux) stage_keys(ks + ks2, key + A.aux_key + (long long)y * N, (long long)kAux * N, L);
        if (staged != sc) {
            if (f64) stage_twiddles(tc, (const double2*)A.tw_fwd_f64 + ((size_t)i << A.logN), m0 + sc);
            else stage_twiddles((ulonglong2*)tc, (const ulonglong2*)A.tw_fwd_int + ((size_t)i << A.logN), m0 + sc);
        }
        staged = sc;
        if (INV && z == 0 && last) {
            if (f64) stage_inverse_twiddles(tc + 256, (const double2*)A.tw_inv_f64 + ((size_t)i << A.logN), m0 + t);
            else stage_inverse_twiddles((ulonglong2*)tc + 256, (const ulonglong2*)A.tw_inv_int + ((size_t)i << A.logN), m0 + t);
        }
        if (z == 0) chain_wait();
        double x[16];  // binary64 or integer words alike
        if (valid) {
#pragma unroll
            for (int e = 0; e < 16; e++) x[e] = __longlong_as_double((long long)p[j + 16 * e]);
        }
        __syncthreads();
        if (valid && own) {  // canonical words of the transform itself
#pragma unroll
            for (int e = 0; e < 16; e++) {
                const u64 v = (u64)__double_as_longlong(x[e]);
                sb[16 * j + (e ^ j)] = f64 ? (u64)__double_as_longlong(ar.inv_input(v)) : v;
            }
        } else if (valid && f64) {
            chunk_forward(ar, x, tc, sb, j, hmask);
#pragma unroll
            for (int e = 0; e < 16; e++) sb[16 * j + (e ^ j)] = (u64)__double_as_longlong(ar.reduce(x[e]));
        } else if (valid) {
#pragma unroll
            for (int e = 0; e < 16; e++) sb[16 * e + (j ^ e)] = (u64)__double_as_longlong(x[e]);
            if (q < (1ULL << 57)) chunk_forward_int(ArithInt<true>(lc), (const ulonglong2*)tc, sb, j, hmask);
            else chunk_forward_int(ArithInt<false>(lc), (const ulonglong2*)tc, sb, j, hmask);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        for (int m = threadIdx.x; m < 256; m += blockDim.x) {
            int s = m;
            if (k != 1u) {
                const int src = galois_src((t << 8) + m, k, A.logN, 1);
                if (!HANN_CHECK_INDEX((src >> 8) - sc, 1)) continue;
                s = src & 255;
            }
            const u64* xp = buf + swz(s);
            if (f64) for (int st = 0; st < (SHARE ? sets : 1); st++) {
                const u64* kp = ks + (SHARE && st ? ks2 : 0) + s;
                u64* ac = acc + (SHARE && st ? acc2 : 0) + swz(m);
                // exact sums of at most eight products in two binary64 words (acc2_fma), reduced on the FP64 pipe; chains of more
                // than eight primes run one item per CTA and add up several such sums
                double r[IB][2];
#pragma unroll
                for (int b = 0; b < IB; b++) {
                    r[b][0] = z ? __longlong_as_double((long long)ac[b * 512]) : 0.0;
                    r[b][1] = z ? __longlong_as_double((long long)ac[b * 512 + 256]) : 0.0;
                }
                for (int d0 = 0; d0 < L; d0 += 8) {
                    double ah[IB][2], al[IB][2];
#pragma unroll
                    for (int b = 0; b < IB; b++) ah[b][0] = ah[b][1] = kAcc2Start, al[b][0] = al[b][1] = 0;
                    const int d1 = d0 + 8 < L ? d0 + 8 : L;
#pragma unroll 4
                    for (int d = d0; d < d1; d++) {
                        const double k0 = residue_to_f64(kp[d << 9]), k1 = residue_to_f64(kp[(d << 9) + 256]);
#pragma unroll
                        for (int b = 0; b < IB; b++) {
                            const double xv = __longlong_as_double((long long)xp[(b * L + d) << 8]);
                            acc2_fma(ah[b][0], al[b][0], k0, xv);
                            acc2_fma(ah[b][1], al[b][1], k1, xv);
                        }
                    }
#pragma unroll
                    for (int b = 0; b < IB; b++)
#pragma unroll
                        for (int c = 0; c < 2; c++) r[b][c] = ar.reduce(__dadd_rn(r[b][c], ar.acc2_value(ah[b][c], al[b][c], c51)));
                    if (IB > 1) break;
                }
#pragma unroll
                for (int b = 0; b < IB; b++) {
                    ac[b * 512] = (u64)__double_as_longlong(r[b][0]);
                    ac[b * 512 + 256] = (u64)__double_as_longlong(r[b][1]);
                }
            } else {
                const u64* kp = ks + s;
                u64* ac = acc + swz(m);
                u64 hi[IB][2], lo[IB][2];
#pragma unroll
                for (int b = 0; b < IB; b++) hi[b][0] = hi[b][1] = lo[b][0] = lo[b][1] = 0;
#pragma unroll 1
                for (int d = 0; d < L; d++) {
                    const u64 k0 = kp[d << 9], k1 = kp[(d << 9) + 256];
#pragma unroll
                    for (int b = 0; b < IB; b++) {
                        const u64 xv = xp[(b * L + d) << 8];
                        mac128(hi[b][0], lo[b][0], xv, k0);
                        mac128(hi[b][1], lo[b][1], xv, k1);
                    }
                }
#pragma unroll
                for (int b = 0; b < IB; b++)
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        const u64 r = reduce128(hi[b][c], lo[b][c], *lc);
                        u64* a = ac + (b * 2 + c) * 256;
                        *a = z ? addmod(*a, r, q) : r;
                    }
            }
        }
    }
    u64* out = A.u + it0 * 2 * UN + (t << 8);
    if (!last || (SHARE && aux)) {  // every thread stores the sums it made
        for (int m = threadIdx.x; m < 256; m += blockDim.x)
            for (int v = 0; v < 2 * nit; v++) out[v * UN + (long long)i * N + m] = acc[v * 256 + swz(m)];
    }
    if (!last) return;
    // those modulo the special prime or with the auxiliary key set go straight into the inverse pass B' of their chunk
    __syncthreads();
    for (int v = hw; v < 2 * nit; v += blockDim.x >> 4) {
        u64* sv = acc + acc2 + v * 256;
        u64* o = out + v * UN + (long long)(L + (aux ? y : 0)) * N;
        const double2* twf = INV ? tc + 256 : (const double2*)A.tw_inv_f64 + ((size_t)i << A.logN);
        const ulonglong2* twi = INV ? (const ulonglong2*)tc + 256 : (const ulonglong2*)A.tw_inv_int + ((size_t)i << A.logN);
        if (f64) chunk_inverse<INV>(ar, twf, m0 + t, sv, o, j, hmask);
        else chunk_inverse<INV>(ArithInt<false>(lc), twi, m0 + t, sv, o, j, hmask);
    }
}

struct HoistArgs {
    const u64* digits;  // pass-A output of digit j for modulus i: (j * L + target of i) * N, a digit's own modulus left out
    const u64* own;     // the polynomial being switched, transform domain, [L][N]
    const u64* const* keytab;
    int rot0, per;      // item `it` is rotation rot0 + it; items per CTA
    long long items;
    u64* u;  // [item][2][L+1][N] as k_ks_apply leaves it, the automorphism still to be applied
    int N, logN;
    const void *tw_fwd_f64, *tw_fwd_int, *tw_inv_f64, *tw_inv_int;
    const LimbConst* lt;
};

// u[item][c][i] = sum_j digit(j) * key_item[j][c] modulo i = L - blockIdx.y, chunk blockIdx.x: one digit set under many keys (hoisted
// rotations).  The CTA runs the second half of the digits' forward transforms on its chunk, then a thread keeps its position's L digit
// words in registers and streams the keys of its items past them, the next item's words in flight.  The special prime's products, eight
// items at a time, meet in shared memory, where the sixteen half-warps run their inverse pass B'.
//
// Bound: HBM, 20 MiB of key and 5 MiB of products per rotation at N = 2^16, L = 4; the special prime's integer transforms (its CTAs
// start first) run beside the stream.  31 rotations: 181 us, in place of 12 (pass B of the digits) + 150 (products) + 50 (inverse pass B').
// Chains of more than four primes keep those three launches: the words of eight digits and of the next item's keys do not fit the
// registers, and read from shared memory and memory in turn they lost (membership circuit 7285 -> 7579 us).
template <int L>
__global__ void __launch_bounds__(256, 3) k_ks_hoist(HoistArgs A) {
    extern __shared__ __align__(16) u64 sm[];
    const int N = A.N, t = blockIdx.x, i = L - (int)blockIdx.y;
    const long long L1N = (long long)(L + 1) * N;
    double2* tc = (double2*)sm;            // [256] forward, [256] inverse
    u64* buf = sm + 1024;                  // [L][256] digits
    u64* acc = buf + (size_t)L * 256;      // [8 items][2][256] products modulo the special prime
    const int it0 = blockIdx.z * A.per, it1 = it0 + A.per < A.items ? it0 + A.per : (int)A.items;
    const int hw = threadIdx.x >> 4, j = threadIdx.x & 15, m = threadIdx.x;
    const unsigned hmask = 0xFFFFu << (threadIdx.x & 16), m0 = (unsigned)(N >> 8);
    const LimbConst* lc = A.lt + i;
    const u64 q = lc->q;
    const bool f64 = q < (1ULL << 50);
    const ArithF64 ar(lc);
    if (f64) stage_twiddles(tc, (const double2*)A.tw_fwd_f64 + ((size_t)i << A.logN), m0 + t);
    else stage_twiddles((ulonglong2*)tc, (const ulonglong2*)A.tw_fwd_int + ((size_t)i << A.logN), m0 + t);
    if (i == L && f64) stage_inverse_twiddles(tc + 256, (const double2*)A.tw_inv_f64 + ((size_t)i << A.logN), m0 + t);
    else if (i == L) stage_inverse_twiddles((ulonglong2*)tc + 256, (const ulonglong2*)A.tw_inv_int + ((size_t)i << A.logN), m0 + t);
    chain_wait();
    __syncthreads();
    for (int dj = hw; dj < L; dj += 16) {
        const bool own = dj == i;
        const u64* p = (own ? A.own + (long long)i * N : A.digits + ((long long)dj * L + (i < dj ? i : i - 1)) * N) + (t << 8);
        u64* sb = buf + dj * 256;
        double x[16];  // binary64 or integer words alike
#pragma unroll
        for (int e = 0; e < 16; e++) x[e] = __longlong_as_double((long long)p[j + 16 * e]);
        if (own) {
#pragma unroll
            for (int e = 0; e < 16; e++) {
                const u64 v = (u64)__double_as_longlong(x[e]);
                sb[16 * j + (e ^ j)] = f64 ? (u64)__double_as_longlong(ar.inv_input(v)) : v;
            }
        } else if (f64) {
            chunk_forward(ar, x, tc, sb, j, hmask);
#pragma unroll
            for (int e = 0; e < 16; e++) sb[16 * j + (e ^ j)] = (u64)__double_as_longlong(ar.reduce(x[e]));
        } else {
#pragma unroll
            for (int e = 0; e < 16; e++) sb[16 * e + (j ^ e)] = (u64)__double_as_longlong(x[e]);
            if (q < (1ULL << 57)) chunk_forward_int(ArithInt<true>(lc), (const ulonglong2*)tc, sb, j, hmask);
            else chunk_forward_int(ArithInt<false>(lc), (const ulonglong2*)tc, sb, j, hmask);
        }
    }
    __syncthreads();
    const u64* xp = buf + swz(m);
    const long long word = (long long)i * N + (t << 8) + m;
    u64* out = A.u + word;
    u64 xd[L];
#pragma unroll
    for (int d = 0; d < L; d++) xd[d] = xp[d << 8];
    u64 cur[2 * L], nxt[2 * L];
    const auto load = [&](int it, u64(&v)[2 * L]) {
        const u64* key = A.keytab[A.rot0 + it] + word;
#pragma unroll
        for (int d = 0; d < 2 * L; d++) v[d] = __ldcs(key + d * L1N);
    };
    // the two sums of an item: balanced binary64 integers below 2^50, residues otherwise
    const auto products = [&](u64(&r)[2]) {
        if (f64) {
            double ah[2] = {kAcc2Start, kAcc2Start}, al[2] = {0, 0};
#pragma unroll
            for (int d = 0; d < L; d++)
#pragma unroll
                for (int c = 0; c < 2; c++) acc2_fma(ah[c], al[c], residue_to_f64(cur[2 * d + c]), __longlong_as_double((long long)xd[d]));
            const double2 c51 = make_double2(lc->c51_bal, lc->c51_q);
#pragma unroll
            for (int c = 0; c < 2; c++) r[c] = (u64)__double_as_longlong(ar.reduce(ar.acc2_value(ah[c], al[c], c51)));
        } else {
            u64 hi[2] = {0, 0}, lo[2] = {0, 0};
#pragma unroll
            for (int d = 0; d < L; d++)
#pragma unroll
                for (int c = 0; c < 2; c++) mac128(hi[c], lo[c], xd[d], cur[2 * d + c]);
            r[0] = reduce128(hi[0], lo[0], *lc);
            r[1] = reduce128(hi[1], lo[1], *lc);
        }
    };
    if (it0 < it1) load(it0, cur);
    for (int b0 = it0; b0 < it1; b0 += 8) {
        const int nb = it1 - b0 < 8 ? it1 - b0 : 8;
#pragma unroll 1
        for (int b = 0; b < nb; b++) {
            const int it = b0 + b;
            if (it + 1 < it1) load(it + 1, nxt);
            u64 r[2];
            products(r);
#pragma unroll
            for (int c = 0; c < 2; c++) {
                if (i < L) out[(long long)(it * 2 + c) * L1N] = r[c];
                else acc[(b * 2 + c) * 256 + swz(m)] = r[c];
            }
#pragma unroll
            for (int d = 0; d < 2 * L; d++) cur[d] = nxt[d];
        }
        if (i < L) continue;
        __syncthreads();
        if (hw < 2 * nb) {
            u64* o = A.u + (long long)(b0 * 2 + hw) * L1N + (long long)i * N + (t << 8);
            u64* sv = acc + hw * 256;
            if (f64) chunk_inverse<true>(ar, tc + 256, m0 + t, sv, o, j, hmask);
            else chunk_inverse<true>(ArithInt<false>(lc), (const ulonglong2*)tc + 256, m0 + t, sv, o, j, hmask);
        }
        __syncthreads();  // the products of the next items may be written
    }
}

struct FinishArgs {
    const u64* lifted;  // [item][2][limbs][N], pass-A format
    const u64* u;       // [item][2] polynomials u_poly words apart; u_mid: binary64 words of limbs below 2^50 (see ApplyArgs)
    long long u_poly;
    int u_mid, limbs;   // limbs of the result
    int last;           // 1: divided by the chain's last prime instead of the special prime
    const u64* add;     // optional: add + item * add_it + component * L N, in the order of the result
    long long add_it;
    const u64* c0;      // optional, first component only: the sum over z of phi_z(c0 + item * c0_it + z * c0_z)
    long long c0_it, c0_z;
    int rot0, rot_inc, nz;  // rotation of z; with PERM, of the item
    u64 *out0, *out1;
    long long out_it;
    u64* next;          // NEXT: inverse pass B' of the second component, [item][limbs][N] (private format)
    const unsigned* galois;
    long long units;    // polynomials: two per item
    int N, logN, n;
    const void *tw_fwd_f64, *tw_fwd_int, *tw_inv_f64, *tw_inv_int;
    const LimbConst* lt;
};

// out[item][c][i] = (u - lifted) d^{-1} + add + phi(c0), d the special prime or the chain's last, modulus i = blockIdx.y, chunk
// blockIdx.x, a half-warp per (item, component): pass B of the lifted ModDown polynomials with the combination behind its last round.
// PERM: u, lifted and c0 are still in the order before the automorphism, which differs from item to item (hoisted rotations); the
// finished words are permuted in shared memory and stored to the item's own chunk of the result.
// NEXT: the result's second component is what the next key switch decomposes, and the half-warp that made a chunk of it runs the
// chunk's inverse pass B' as well: a launch and two passes over the polynomial less for every step of a chain of key switches.
//
// 31 rotations at N = 2^16, L = 4: 170 us (pass B and the combination as two kernels) -> 103 us; the integer reductions of the
// combination and a 16-fold unrolled tail (instruction fetch) cost most of that on the way.
template <bool PERM, bool NEXT>
__global__ void __launch_bounds__(256, 3) k_ks_finish(FinishArgs A) {
    extern __shared__ __align__(16) u64 sm[];
    const int N = A.N, t = blockIdx.x, i = blockIdx.y;
    const long long LN = (long long)A.limbs * N;
    double2* tc = (double2*)sm;
    const int hw = threadIdx.x >> 4, j = threadIdx.x & 15;
    const unsigned hmask = 0xFFFFu << (threadIdx.x & 16);
    u64* sb = sm + 512 + hw * 256;
    const LimbConst* lc = A.lt + i;
    const u64 q = lc->q;
    const unsigned m0 = (unsigned)(N >> 8);
    const bool f64 = q < (1ULL << 50);
    const ArithF64 ar(lc);
    const double2 pinv = A.last ? make_double2(lc->linv_bal, lc->linv_q) : make_double2(lc->pinv_bal, lc->pinv_q);
    const u64 pinv_i = A.last ? lc->linv : lc->pinv, pinv_s = A.last ? lc->linv_s : lc->pinv_s;
    if (f64) stage_twiddles(tc, (const double2*)A.tw_fwd_f64 + ((size_t)i << A.logN), m0 + t);
    else stage_twiddles((ulonglong2*)tc, (const ulonglong2*)A.tw_fwd_int + ((size_t)i << A.logN), m0 + t);
    chain_wait();
    __syncthreads();
    const long long units = A.units, ustep = (long long)gridDim.z * (blockDim.x >> 4);
    for (long long k = (long long)blockIdx.z * (blockDim.x >> 4) + hw; k < units; k += ustep) {
        // (NEXT: second components after all first ones, so that the half-warps of a warp do the same)
        const long long items = units >> 1, v = !NEXT ? k : k < items ? 2 * k : 2 * (k - items) + 1;
        const long long item = v >> 1;
        const int c = (int)(v & 1);
        const u64* p = A.lifted + (v * A.limbs + i) * N + (t << 8);
        const u64* up = A.u + v * A.u_poly + (long long)i * N + (t << 8) + j;
        const u64* ap = A.add ? A.add + item * A.add_it + c * LN + (long long)i * N + (t << 8) + j : nullptr;
        const u64* cp = A.c0 && c == 0 ? A.c0 + item * A.c0_it + (long long)i * N : nullptr;
        u64* o = (c == 0 ? A.out0 : A.out1) + item * A.out_it + (long long)i * N;
        double x[16];
#pragma unroll
        for (int e = 0; e < 16; e++) x[e] = __longlong_as_double((long long)p[j + 16 * e]);
        __syncwarp(hmask);  // the words of the half-warp's previous polynomial have been taken
        // then words 16 e + j, eight at a time: the combination is long and a rolled loop keeps its instructions few
        if (f64) {
            chunk_forward(ar, x, tc, sb, j, hmask);
#pragma unroll
            for (int e = 0; e < 16; e++) sb[16 * j + (e ^ j)] = (u64)__double_as_longlong(ar.reduce(x[e]));
#pragma unroll 1
            for (int e0 = 0; e0 < 16; e0 += 8) {
                double uw[8], a[8];
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    const u64 v = up[16 * (e0 + e)];
                    uw[e] = A.u_mid ? ar.from_mid(v) : ar.from_canonical(v);
                }
#pragma unroll
                for (int e = 0; e < 8; e++) a[e] = ap ? ar.from_canonical(ap[16 * (e0 + e)]) : 0.0;
                if (PERM && cp) {
#pragma unroll
                    for (int e = 0; e < 8; e++) a[e] = ar.from_canonical(cp[(t << 8) + 16 * (e0 + e) + j]);
                } else if (cp) {
                    for (int z = 0; z < A.nz; z++) {
                        const LaneSource ls((t << 8) + j, A.galois[A.rot0 + z * A.rot_inc], A.logN);
#pragma unroll
                        for (int e = 0; e < 8; e++) {
                            const int w = ls.word(e0 + e);
                            if (!HANN_CHECK_INDEX(w, N)) continue;
                            a[e] = __dadd_rn(a[e], ar.from_canonical(cp[z * A.c0_z + w]));
                            if ((z & 3) == 3) a[e] = ar.reduce(a[e]);
                        }
                    }
                }
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    // |u - reduce(x)| <= 1.5 q, the product lies below 0.7 q, the added words below 5 q
                    u64* w = sb + 16 * j + ((e0 + e) ^ j);
                    const double y = ar.mulmod_small(__dsub_rn(uw[e], __longlong_as_double((long long)*w)), pinv);
                    double v = __dadd_rn(y, a[e]);
                    if (NEXT) {
                        v = ar.reduce(v);
                        *w = (u64)__double_as_longlong(v);
                    }
                    const u64 r = ar.to_canonical(v);
                    if (PERM) *w = r;
                    else o[(t << 8) + 16 * (e0 + e) + j] = r;
                }
            }
        } else {
#pragma unroll
            for (int e = 0; e < 16; e++) sb[16 * e + (j ^ e)] = (u64)__double_as_longlong(x[e]);
            if (q < (1ULL << 57)) chunk_forward_int(ArithInt<true>(lc), (const ulonglong2*)tc, sb, j, hmask);
            else chunk_forward_int(ArithInt<false>(lc), (const ulonglong2*)tc, sb, j, hmask);
#pragma unroll 2
            for (int e = 0; e < 16; e++) {
                u64* w = sb + 16 * j + (e ^ j);
                u64 r = csub(shoup_mul(submod(up[16 * e], *w, q), pinv_i, pinv_s, q), q);
                if (ap) r = addmod(r, ap[16 * e], q);
                if (PERM && cp) {
                    r = addmod(r, cp[(t << 8) + 16 * e + j], q);
                } else if (cp) {
                    for (int z = 0; z < A.nz; z++) {
                        const int src = galois_src((t << 8) + 16 * e + j, A.galois[A.rot0 + z * A.rot_inc], A.logN, 1);
                        if (!HANN_CHECK_INDEX(src, N)) continue;
                        r = addmod(r, cp[z * A.c0_z + src], q);
                    }
                }
                if (PERM || NEXT) *w = r;
                if (!PERM) o[(t << 8) + 16 * e + j] = r;
            }
        }
        if (NEXT && c == 1) {
            u64* nx = A.next + item * LN + (long long)i * N + (t << 8);
            if (f64) chunk_inverse<false>(ar, (const double2*)A.tw_inv_f64 + ((size_t)i << A.logN), m0 + t, sb, nx, j, hmask);
            else chunk_inverse<false>(ArithInt<false>(lc), (const ulonglong2*)A.tw_inv_int + ((size_t)i << A.logN), m0 + t, sb, nx, j, hmask);
        }
        if (PERM) {
            const int r = A.rot0 + (int)item * A.rot_inc;
            const unsigned k = A.galois[r], kinv = A.galois[(A.n - r) % A.n];
            const int tt = galois_src(t << 8, kinv, A.logN, 1) >> 8;  // the chunk of the result that reads this one
            const LaneSource ls((tt << 8) + j, k, A.logN);
            const bool inside = HANN_CHECK_INDEX((ls.base >> 8) - t, 1);
            const u64* sr = sb + ((ls.base & 15) << 4);  // logical position 16 a + b at word 16 a + (b ^ a), a the word's low nibble
            __syncwarp(hmask);
#pragma unroll 8
            for (int e = 0; e < 16; e++)
                if (inside) o[(tt << 8) + 16 * e + j] = sr[ls.high(e) ^ (ls.base & 15)];
        }
    }
}

int run_finish(hann_ctx* c, FinishArgs& A, bool perm_items) {
    A.galois = c->galois_dev;
    A.N = c->N;
    A.logN = c->logN;
    A.n = c->n;
    A.tw_fwd_f64 = c->tw_fwd_f64;
    A.tw_fwd_int = c->tw_fwd;
    A.tw_inv_f64 = c->tw_inv_f64;
    A.tw_inv_int = c->tw_inv;
    A.lt = c->lt_dev;
    // up to sixteen half-warps per CTA, which then walk further polynomials under the staged tables while the grid fills the
    // machine twice over
    const int hws = (int)(A.units < 16 ? A.units : 16), threads = (16 * hws + 31) / 32 * 32;
    const size_t smem = 4096 + (size_t)threads / 16 * 2048;
    const long long per = (long long)(c->N >> 8) * A.limbs, groups = (A.units + threads / 16 - 1) / (threads / 16);
    long long gz = (2 * 148 * 3 + per - 1) / per;
    if (gz > groups) gz = groups;
    KProf kp(c, KC_MODDOWN_COMBINE);
    const auto kern = perm_items ? k_ks_finish<true, false> : A.next ? k_ks_finish<false, true> : k_ks_finish<false, false>;
    launch_chain(c, kern, dim3(c->N >> 8, A.limbs, (unsigned)gz), threads, smem, A);
    return check_launch(c, "ks_finish");
}

// sixteen lanes per digit, whole warps
constexpr int apply_threads(int IB, int L) { return (IB * L * 16 + 31) / 32 * 32; }
constexpr size_t apply_smem(int IB, int L, bool share = false, bool inv = true) {
    return (inv ? 8192 : 4096) + (size_t)((share ? 2 : 1) * (2 * L + 2 * IB) + apply_threads(IB, L) / 16) * 2048;
}

constexpr size_t hoist_smem(int L) { return 8192 + (size_t)(L + 16) * 2048; }

template <int IB, int T, bool SHARE = false>
void launch_apply(hann_ctx* c, const ApplyArgs& A) {
    KProf kp(c, KC_KS_INNER);
    launch_chain(c, k_ks_apply<IB, T, SHARE>, dim3(c->N >> 8, SHARE ? A.L : A.L + A.nx, (unsigned)((A.items + IB - 1) / IB)), apply_threads(IB, A.L),
                 apply_smem(IB, A.L, SHARE, T >= 256), A);
}

}  // namespace

// Dynamic shared memory of the instances that may need more than the default 48 KiB, for the longest chain launch_ks_apply sends to
// each.  The limit belongs to the kernel and the device, not to a context: it is the same for every context, so that contexts of
// different chain lengths do not take it from one another.
int ks_fused_configure() {
    static_assert(apply_smem(2, 4, false, false) <= 48 * 1024 && apply_smem(1, 4, false, false) <= 48 * 1024, "the other instances need no opt-in");
    if (cudaFuncSetAttribute(k_ks_apply<4, 256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)apply_smem(4, 4)) != cudaSuccess) return HANN_ECUDA;
    if (cudaFuncSetAttribute(k_ks_apply<4, 256, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)apply_smem(4, 4, true)) != cudaSuccess) return HANN_ECUDA;
    if (cudaFuncSetAttribute(k_ks_apply<2, 256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)apply_smem(2, 8)) != cudaSuccess) return HANN_ECUDA;
    if (cudaFuncSetAttribute(k_ks_apply<1, 256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)apply_smem(1, HANN_MAX_PRIMES)) != cudaSuccess)
        return HANN_ECUDA;
    static_assert(hoist_smem(4) <= 48 * 1024, "k_ks_hoist needs no opt-in");
    return HANN_OK;
}

bool ks_fused_available(const hann_ctx* c) { return c->logN >= 10 && c->ntt_tau; }
bool ks_hoist_available(const hann_ctx* c) { return ks_fused_available(c) && c->L <= 4; }

// digits: output of launch_ks_lift for the nz * items polynomials of L limbs; own (optional): the polynomials themselves, in which
// case the digits were lifted without their own modulus.  aux (only with own): they were lifted without the special prime as well, and
// every key of the launch has its auxiliary words.
// Leaves u[item][2][L + nx][N] (see ApplyArgs), the input of the ModDown lift.
int launch_ks_apply(hann_ctx* c, const u64* digits, const u64* own, int64_t own_it, int64_t own_z, int64_t items, int nz, int rot0, int rot_zinc, bool aux, u64* u) {
    if (items <= 0 || nz <= 0) return HANN_OK;
    ApplyArgs A = {};
    A.digits = digits;
    A.nx = aux ? kAux : 1;
    for (int k = 0; k < kAux; k++) A.aux4 |= (u64)c->crt.limb[k] << (4 * k);
    for (int l = 0, k = kAux; aux && l < c->L; l++)
        if (l != c->crt.limb[0] && l != c->crt.limb[1] && l != c->crt.limb[2]) A.aux4 |= (u64)l << (4 * k++);
    A.aux_key = (long long)c->L * 2 * (c->L + 1) * c->N;
    A.n_tgt = aux ? c->L - 1 : own ? c->L : c->L + 1;
    A.own = own;
    A.own_it = own_it;
    A.own_z = own_z;
    A.keytab = c->keytab_dev;
    A.galois = c->galois_dev;
    A.rot0 = rot0;
    A.rot_zinc = rot_zinc;
    A.nz = nz;
    A.items = items;
    A.u = u;
    A.N = c->N;
    A.logN = c->logN;
    A.L = c->L;
    A.tw_fwd_f64 = c->tw_fwd_f64;
    A.tw_fwd_int = c->tw_fwd;
    A.tw_inv_f64 = c->tw_inv_f64;
    A.tw_inv_int = c->tw_inv;
    A.lt = c->lt_dev;
    // Items per CTA: their digits fill at most sixteen half-warps, and the eight-product sums allow several items up to eight
    // primes only; key words and table entries are read once for all of them.  Us of a launch with one / two / four items per CTA
    // (the absent items of a ragged last CTA cost their products all the same):
    //   N = 2^16, L = 4, one rotation:    1 item 22 / 24 / 38, 2: 37 / 31 / 42, 3: 54 / 48 / 50, 4: 69 / 52 / 52, 5: 85 / 70 / 86, 8: 131 / 100 / 98
    //             three rotations:        1 item 52 / 65 / 100, 2: 92 / 73 / 106, 4: 173 / 129 / 130, 5: 212 / 177 / 215, 16: 646 / 468 / 472
    //   N = 2^15, L = 4, one rotation:    1 item 18 / 19 / 22, 2: 23 / 21 / 23, 4: 43 / 33 / 28, 8: 77 / 57 / 51, 16: 140 / 105 / 96
    //   N = 2^12, L = 2, seven rotations: 1 item 78 / 68 / 62, 16: 86 / 88 / 83
    //   N = 2^15, L = 8, one rotation:    1 item 24 / 32, 2: 45 / 42, 3: 64 / 70, 4: 82 / 77, 16: 292 / 281
    // (taken with the special prime itself).  Four items of five or six leave most of the last CTA empty.  Us of the launches of a call with
    // three giant steps, two / four items per CTA (aux: with auxiliary primes, whose key set four items take from the same transforms):
    //   N = 2^16, L = 4, aux:  Horner, 4 blocks 456 / 441, 5 566 / 572, 6 607 / 606, 8 758 / 713   lazy, 4 273 / 251, 5 348 / 348
    //             without:     Horner, 4 blocks 460 / 472, 5 552 / 602, 6 604 / 643, 8 747 / 750   lazy, 5 352 / 392
    //   N = 2^15, L = 4, aux:  Horner, 5 345 / 347, 6 358 / 357      without: 5 338 / 350, 6 350 / 362, 7 422 / 412
    //   N = 2^16, L = 3, aux:  Horner, 4 351 / 347, 5 471 / 493, 6 491 / 508     without: 5 469 / 508, 6 489 / 523, 7 552 / 566
    //   N = 2^15, L = 3, aux:  Horner, 5 288 / 295, 6 301 / 309      without: 5 294 / 301, 6 309 / 312, 7 352 / 340
    //   N = 2^16, L = 2:       Horner, 5 364 / 353, 6 368 / 360      N = 2^15, L = 2: 5 232 / 226, 6 234 / 232
    const bool ragged = (items == 5 || items == 6) && (c->L == 3 || (c->L == 4 && !aux));
    if (items >= 4 && !ragged && c->L <= 4 && aux) launch_apply<4, 256, true>(c, A);
    else if (items >= 4 && !ragged && c->L <= 4) launch_apply<4, 256>(c, A);
    else if (items >= 2 && c->L <= 4) launch_apply<2, 128>(c, A);
    else if (items >= 2 && c->L <= 8) launch_apply<2, 256>(c, A);
    else if (c->L <= 4) launch_apply<1, 64>(c, A);
    else launch_apply<1, 256>(c, A);
    return check_launch(c, "ks_apply");
}

// digits: output of launch_ks_lift for one polynomial of L limbs, own, whose digits were lifted without their own modulus.  Leaves
// u[item][2][L+1][N], item `it` under the key of rotation rot0 + it, for the ModDown lift and launch_ks_finish with perm_items.  Only where
// ks_hoist_available(c) holds.
int launch_ks_hoist(hann_ctx* c, const u64* digits, const u64* own, int64_t items, int rot0, u64* u) {
    if (items <= 0) return HANN_OK;
    HoistArgs A = {};
    A.digits = digits;
    A.own = own;
    A.keytab = c->keytab_dev;
    A.rot0 = rot0;
    A.items = items;
    A.u = u;
    A.N = c->N;
    A.logN = c->logN;
    A.tw_fwd_f64 = c->tw_fwd_f64;
    A.tw_fwd_int = c->tw_fwd;
    A.tw_inv_f64 = c->tw_inv_f64;
    A.tw_inv_int = c->tw_inv;
    A.lt = c->lt_dev;
    // CTAs that share out the items of a chunk: smallest (waves x items of a CTA, the digits counting as two), ties to fewer; no less
    // than the CTAs of the special prime take, an item of which is two (products and inverse passes).  Without that bound a launch below
    // one wave took one CTA a chunk and lasted as long as those (us of a level of 1000 rows, L = 2, R = 128, B = 32, 1 / 2 / 3 / 4 / 8 CTAs:
    // N = 2^15 293 / 260 / 265 / 264 / 274, N = 2^14 198 / 184 / 182 / 180 / 185; L = 4, N = 2^16, five waves: 692 / 695 / 706 / 711 / 755).
    const long per = (long)(c->N >> 8) * (c->L + 1), slots = 148 * 3;
    int gz = 1;
    long best = -1;
    for (int z = 1; z <= items && z <= 64; z++) {
        const long n = (items + z - 1) / z, cost = std::max(((per * z + slots - 1) / slots) * (2 + n), 2 + 2 * n);
        if (best < 0 || cost < best) {
            best = cost;
            gz = z;
        }
    }
    A.per = (int)((items + gz - 1) / gz);
    KProf kp(c, KC_KS_INNER_KEYS);
    auto go = [&](auto kern) { launch_chain(c, kern, dim3(c->N >> 8, c->L + 1, (unsigned)((items + A.per - 1) / A.per)), 256, hoist_smem(c->L), A); };
    switch (c->L) {
        case 1: go(k_ks_hoist<1>); break;
        case 2: go(k_ks_hoist<2>); break;
        case 3: go(k_ks_hoist<3>); break;
        default: go(k_ks_hoist<4>); break;
    }
    return check_launch(c, "ks_hoist");
}

// lifted: output of launch_ks_lift (launch_ks_lift_aux) for the special-prime (auxiliary) limbs of u, whose polynomials have u_limbs
// limbs.  perm_items: the automorphism is still to be applied, that of item `it` being rotation rot0 + it * rot_inc (otherwise rotation
// rot0 + z * rot_inc belongs to the c0 term z < nz).  next (optional, not with perm_items): the second components after their inverse
// pass B', [item][L][N], for a key switch that follows.
int launch_ks_finish(hann_ctx* c, const u64* u, int u_limbs, const u64* lifted, int64_t items, bool perm_items, int rot0, int rot_inc, int nz,
                     const u64* c0, int64_t c0_it, int64_t c0_z, const u64* add, int64_t add_it, u64* out0, u64* out1, int64_t out_it, u64* next) {
    if (items <= 0) return HANN_OK;
    FinishArgs A = {};
    A.lifted = lifted;
    A.u = u;
    A.u_poly = (long long)u_limbs * c->N;
    A.u_mid = perm_items && !ks_hoist_available(c) ? 0 : 1;
    A.limbs = c->L;
    A.add = add;
    A.add_it = add_it;
    A.c0 = c0;
    A.c0_it = c0_it;
    A.c0_z = c0_z;
    A.rot0 = rot0;
    A.rot_inc = rot_inc;
    A.nz = nz;
    A.out0 = out0;
    A.out1 = out1;
    A.out_it = out_it;
    A.next = next;
    A.units = 2 * items;
    return run_finish(c, A, perm_items);
}

// out[poly][i] = (src[poly][i] - lifted[poly][i]) q_{L-1}^{-1}, i < keep; src polynomials have L limbs.  One launch in place of pass B
// and a combination, and the lift in place of an inverse pass A, a lift and a pass A.
int launch_rescale_finish(hann_ctx* c, const u64* src, const u64* lifted, int64_t npoly, int keep, u64* out) {
    if (npoly <= 0) return HANN_OK;
    FinishArgs A = {};
    A.lifted = lifted;
    A.u = src;
    A.u_poly = (long long)c->L * c->N;
    A.limbs = keep;
    A.last = 1;
    A.out0 = out;
    A.out1 = out + (int64_t)keep * c->N;
    A.out_it = 2 * (int64_t)keep * c->N;
    A.units = npoly;
    return run_finish(c, A, false);
}

HANN_DEBUG_DEFINE_BIND(debug_bind_ksfused)
