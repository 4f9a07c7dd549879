// The client's decode on the device: residues of a decrypted polynomial -> centred integers (CRT) -> binary64 -> twist and inverse
// canonical embedding (a complex FFT) -> slot values.
//
// A coefficient's residues become mixed-radix digits (Garner), those a multi-word integer, which is centred against Q/2, multiplied by
// a small integer (a rescaled ciphertext's scale is 2^k / q) and rounded to binary64 ONCE, to nearest even, before the exact scaling by a
// power of two: no intermediate of fewer digits, whatever the chain's length.  The FFT is the radix-2 decimation-in-time graph of the
// encoder with conjugated, correctly rounded twiddles, every product and sum rounded separately.
//
// On the host (long double Garner and FFT, one ciphertext after the other) the 7 ciphertexts of 222,049 rows took 45 ms of a 48 ms
// decryption; here the kernels take 0.17 ms (CRT 27 us, FFT 25 us, transforms the rest) beside 1.2 ms of copies.
#include "internal.h"

namespace {

constexpr int kThreads = 256;

struct CrtConst {
    u64 inv[HANN_MAXL1 - 1][HANN_MAXL1 - 1];  // inv[i][k] = q_k^{-1} mod q_i, k < i
    u64 Q[HANN_MAXL1], half[HANN_MAXL1];      // product of the primes and its half (rounded down), least significant word first
};

// magnitude w (NW words) with sign -> nearest binary64
template <int NW>
__device__ __forceinline__ double round_to_f64(const u64 (&w)[NW], bool neg) {
    u64 top = 0, next = 0;
    bool sticky = false;
    int e = 0;
#pragma unroll
    for (int i = 0; i < NW; i++) {  // from the least significant word: top takes the last non-zero one
        if (w[i]) {
            sticky = sticky || next != 0;
            next = i > 0 ? w[i > 0 ? i - 1 : 0] : 0;
            top = w[i];
            e = 64 * i;
        }
    }
    // words below `next` that are non-zero but were not seen as a predecessor of a non-zero word
#pragma unroll
    for (int i = 0; i < NW; i++) sticky = sticky || (64 * (i + 1) < e && w[i] != 0);
    if (!top) return 0.0;
    const int sh = __clzll((long long)top);
    if (sh) {
        top = (top << sh) | (next >> (64 - sh));
        next <<= sh;
    }
    const u64 m = top | (sticky || next ? 1 : 0);  // 64 bits, the lowest one sticky: the conversion below rounds the whole number
    const double d = scalbn(__ull2double_rn(m), e - sh);
    return neg ? -d : d;
}

// one coefficient: residues r[i] (canonical) -> nearest binary64 of mult * (the centred integer modulo the product of the L primes)
template <int NW>  // words of the largest product (L <= NW - 1)
__device__ __forceinline__ double crt_value(const u64 (&r)[NW - 1], int L, u64 mult, const CrtConst& cc, const LimbTable& lt) {
    u64 v[NW - 1];
#pragma unroll
    for (int i = 0; i < NW - 1; i++) {
        if (i < L) {
            const LimbConst& lc = lt.c[i];
            u64 t = r[i];
#pragma unroll
            for (int k = 0; k < i; k++) t = mulmod(submod(t, barrett64(v[k], lc), lc.q), cc.inv[i][k], lc);
            v[i] = t;
        }
    }
    u64 x[NW];
#pragma unroll
    for (int i = 0; i < NW; i++) x[i] = 0;
    auto mul_add = [&](u64 m, u64 a) {  // x = x * m + a
#pragma unroll
        for (int i = 0; i < NW; i++) {
            const u64 lo = x[i] * m, hi = __umul64hi(x[i], m);
            x[i] = lo + a;
            a = hi + (x[i] < lo ? 1 : 0);
        }
    };
#pragma unroll
    for (int i = NW - 2; i >= 0; i--)
        if (i < L) mul_add(lt.c[i].q, v[i]);  // v_0 + q_0 (v_1 + q_1 (v_2 + ..))
    bool neg = false, decided = false;
#pragma unroll
    for (int i = NW - 1; i >= 0; i--) {
        const u64 h = i < HANN_MAXL1 ? cc.half[i < HANN_MAXL1 ? i : 0] : 0;
        if (!decided && x[i] != h) {
            neg = x[i] > h;
            decided = true;
        }
    }
    if (neg) {
        u64 borrow = 0;
#pragma unroll
        for (int i = 0; i < NW; i++) {
            const u64 a = i < HANN_MAXL1 ? cc.Q[i < HANN_MAXL1 ? i : 0] : 0, d = a - x[i], d2 = d - borrow;
            borrow = (a < x[i] || d < borrow) ? 1 : 0;
            x[i] = d2;
        }
    }
    if (mult != 1) mul_add(mult, 0);
    return round_to_f64<NW>(x, neg);
}

// mu = c0 + prod modulo each prime (c0 canonical or not, prod canonical) -> buf[P][brev(k)] = (m_k + i m_{k+n}) conj(U_k), m scaled
template <int NW>
__global__ void __launch_bounds__(128) k_decode_crt(const u64* __restrict__ c0, const u64* __restrict__ prod, double2* __restrict__ buf,
                                                    const double2* __restrict__ U, int logn, int L, u64 mult, int exp2, CrtConst cc, LimbTable lt) {
    const int n = 1 << logn, N = 2 * n, k = blockIdx.x * 128 + threadIdx.x;
    if (k >= n) return;
    const long long base = (long long)blockIdx.y * L * N;
    double m[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        u64 r[NW - 1];
#pragma unroll
        for (int i = 0; i < NW - 1; i++)
            if (i < L) {
                const long long o = base + (long long)i * N + k + h * n;
                r[i] = addmod(barrett64(c0[o], lt.c[i]), prod[o], lt.c[i].q);
            }
        m[h] = scalbn(crt_value<NW>(r, L, mult, cc, lt), exp2);
    }
    const double ur = U[k].x, ui = -U[k].y;
    const int pos = (int)(__brev((unsigned)k) >> (32 - logn));
    buf[((long long)blockIdx.y << logn) + pos] = make_double2(__dsub_rn(__dmul_rn(m[0], ur), __dmul_rn(m[1], ui)),
                                                              __dadd_rn(__dmul_rn(m[0], ui), __dmul_rn(m[1], ur)));
}

__device__ __forceinline__ void butterfly_conj(double2& x, double2& y, double2 w) {  // w conjugated: exp(+2 pi i t / n)
    const double vr = __dadd_rn(__dmul_rn(y.x, w.x), __dmul_rn(y.y, w.y)), vi = __dsub_rn(__dmul_rn(y.y, w.x), __dmul_rn(y.x, w.y));
    y = make_double2(__dsub_rn(x.x, vr), __dsub_rn(x.y, vi));
    x = make_double2(__dadd_rn(x.x, vr), __dadd_rn(x.y, vi));
}

// stages 1 .. b1 on contiguous chunks of 2^b1 points, K1 chunks per CTA, in place
__global__ void __launch_bounds__(kThreads) k_decode_fft_a(double2* __restrict__ buf, const double2* __restrict__ T, int logn, int b1, int K1) {
    extern __shared__ double2 smc[];
    const int n = 1 << logn, S1 = 1 << b1, words = K1 * S1;
    double2* p = buf + (long long)blockIdx.y * n + (long long)blockIdx.x * words;
    for (int idx = threadIdx.x; idx < words; idx += kThreads) smc[idx] = p[idx];
    __syncthreads();
    for (int s = 1; s <= b1; s++) {
        const int h = 1 << (s - 1);
        for (int bf = threadIdx.x; bf < words / 2; bf += kThreads) {
            const int t = bf & (h - 1), i0 = ((bf >> (s - 1)) << s) + t;
            butterfly_conj(smc[i0], smc[i0 + h], T[t << (logn - s)]);
        }
        __syncthreads();
    }
    for (int idx = threadIdx.x; idx < words; idx += kThreads) p[idx] = smc[idx];
}

// the remaining stages on C1 columns of the (n / 2^b1) x 2^b1 matrix view; FFT output u goes to slot jpos[brev(u)]
__global__ void __launch_bounds__(kThreads) k_decode_fft_b(const double2* __restrict__ buf, const double2* __restrict__ T, const int32_t* __restrict__ jpos,
                                                           int logn, int b1, int C1, double* __restrict__ re, double* __restrict__ im) {
    extern __shared__ double2 smc[];
    const int n = 1 << logn, S1 = 1 << b1, rows = n >> b1, c0 = blockIdx.x * C1;
    const double2* in = buf + (long long)blockIdx.y * n + c0;
    for (int idx = threadIdx.x; idx < rows * C1; idx += kThreads) smc[idx] = in[(long long)(idx / C1) * S1 + (idx % C1)];
    __syncthreads();
    for (int s = b1 + 1; s <= logn; s++) {
        const int hr = 1 << (s - 1 - b1);
        for (int bf = threadIdx.x; bf < (rows / 2) * C1; bf += kThreads) {
            const int c = bf % C1, rb = bf / C1, tr = rb & (hr - 1), r0 = (rb / hr) * 2 * hr + tr;
            butterfly_conj(smc[r0 * C1 + c], smc[(r0 + hr) * C1 + c], T[(long long)(tr * S1 + c0 + c) << (logn - s)]);
        }
        __syncthreads();
    }
    for (int idx = threadIdx.x; idx < rows * C1; idx += kThreads) {
        const int u = (idx / C1) * S1 + c0 + (idx % C1);
        const long long j = (long long)blockIdx.y * n + jpos[__brev((unsigned)u) >> (32 - logn)];
        re[j] = smc[idx].x;
        if (im) im[j] = smc[idx].y;
    }
}

}  // namespace

// count decrypted polynomials mu = c0 + prod (coefficient domain, [count][L][N], prod canonical) over the first L primes -> real (and
// imaginary, im not null) parts of their slots times mult * 2^exp2, [count][n]; buf: count * n complex numbers
int launch_decode(hann_ctx* c, const u64* c0, const u64* prod, int64_t count, int L, u64 mult, int exp2, double2* buf, double* re, double* im) {
    if (count <= 0) return HANN_OK;
    CrtConst cc = {};
    for (int i = 0; i < L; i++)
        for (int k = 0; k < i; k++) cc.inv[i][k] = hm::invmod(c->mod[k] % c->mod[i], c->mod[i]);
    cc.Q[0] = 1;
    for (int i = 0; i < L; i++) {
        unsigned __int128 carry = 0;
        for (int w = 0; w < HANN_MAXL1; w++) {
            carry += (unsigned __int128)cc.Q[w] * c->mod[i];
            cc.Q[w] = (u64)carry;
            carry >>= 64;
        }
    }
    for (int w = 0; w < HANN_MAXL1; w++) cc.half[w] = (cc.Q[w] >> 1) | (w + 1 < HANN_MAXL1 ? cc.Q[w + 1] << 63 : 0);
    const int n = c->n, logn = c->logN - 1;
    {
        KProf kp(c, KC_OTHER);
        const dim3 grid((n + 127) / 128, (unsigned)count);
        auto go = [&](auto kern) { kern<<<grid, 128, 0, c->stream>>>(c0, prod, buf, c->fft_U, logn, L, mult, exp2, cc, c->lt); };
        // (a chain of L primes below 2^62 and the multiplier fit L + 1 words)
        if (L <= 2) go(k_decode_crt<3>);
        else if (L <= 4) go(k_decode_crt<5>);
        else if (L <= 8) go(k_decode_crt<9>);
        else go(k_decode_crt<HANN_MAXL1>);
    }
    const int b1 = logn < 8 ? logn : 8, S1 = 1 << b1, chunks = n >> b1, K1 = chunks < 8 ? chunks : 8, C1 = S1 < 16 ? S1 : 16;
    {
        KProf kp(c, KC_FFT_A);
        k_decode_fft_a<<<dim3(chunks / K1, (unsigned)count), kThreads, (size_t)K1 * S1 * sizeof(double2), c->stream>>>(buf, c->fft_T, logn, b1, K1);
    }
    {
        KProf kp(c, KC_FFT_B);
        k_decode_fft_b<<<dim3(S1 / C1, (unsigned)count), kThreads, (size_t)(n >> b1) * C1 * sizeof(double2), c->stream>>>(buf, c->fft_T, c->jinv, logn, b1, C1,
                                                                                                                        re, im);
    }
    return check_launch(c, "decode");
}
