// Spectral solution of Poisson's equation (Section III-E, Eqs. 8-12) on FP32
// fast Fourier transforms.
//
// With C(u,x) = cos(pi u (2x+1) / 2n) and S(u,x) = sin(...):
//   a[v][u] = eps_u eps_v / n^2  sum_y sum_x rho[y][x] C(u,x) C(v,y)   (Eq. 10)
//   Psi = a / (w_u^2 + w_v^2), Psi_00 = 0
//   psi[y][x] = sum_u C(u,x) P[u][y],        P[u][y] = sum_v Psi[v][u] C(v,y)
//   E_x[y][x] = sum_u w_u S(u,x) P[u][y]
//   E_y[y][x] = sum_u C(u,x) R[u][y],        R[u][y] = sum_v w_v Psi[v][u] S(v,y)
//
// Three passes:
//   rows_fwd  : rho rows -> DCT-II along x -> T1 (written transposed)
//   cols      : T1 rows  -> DCT-II along y -> divide -> inverse along y for P
//               and R -> PT, RT (written transposed); the energy
//               N = 1/2 A_b sum B Psi (Parseval) is reduced here
//   rows_inv  : PT, RT rows -> E_x, E_y rows (psi from PT on demand)
// The transposed maps hold two neighbouring rows interleaved, as the complex
// rows of the next pass's FFTs: T1[u/2][y] = (u even, u odd) and
// PT[y/2][u], RT[y/2][u] = (y even, y odd).
//
// Each 1-D cosine transform of length n is one complex FFT of length n
// (Makhoul's reordering: v[k] = r[2k], v[n-1-k] = r[2k+1]; A[u] =
// Re(exp(-i pi u / 2n) V[u])), two real rows packed into one complex FFT.
// The inverse cosine sum y[x] = sum_u c[u] C(u,x) is the inverse of that map;
// a sine sum is a cosine sum of the reversed coefficients times (-1)^x.
//
// The FFT lives in registers: n/E threads per FFT hold E elements each.  A
// Stockham FFT of radices n / E^k, E, .., E reads in every stage and leaves
// at the end, in thread t, the elements t + (n/E) q, q < E, whatever the
// radix, so that the work around the FFTs needs no shared memory either:
// Makhoul's order (elements p and n-1-p), the split of two packed spectra
// (u and n-u) and the unshuffle pair element q of thread t with element
// E-1-q of thread n/E-1-t or n/E-t, and the threads are numbered so that this
// is another lane of the same warp (lane_rev, lane_neg): one shuffle.  Only
// the exchanges between stages go through shared memory (two at n = 2048).
// What bounds it: latency and the FP32 pipe.  Against the same transforms
// with every stage, the packing and the unshuffle through shared buffers
// (bound by the shared-memory pipe at 22 % warps active), launch times under
// ncu, cold caches: n = 2048 rows_fwd 19.9 -> 15.2, cols 39.3 -> 24.5,
// rows_inv 26.6 -> 15.8 us; n = 4096 96 -> 58, 187 -> 99, 111 -> 52 us.
#include <type_traits>

#include "fftpl_internal.cuh"

namespace fftpl {

// ------------------------------------- stores through the TMA unit
// A pass that writes its output transposed first lays the tile out in shared
// memory in the output's order, then one thread stores it box by box with
// cp.async.bulk.tensor: the tile leaves the SM as whole 32-byte rows of the
// box instead of one piece per thread and store instruction.
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Every thread that wrote part of a tile: its shared-memory writes become
// visible to the asynchronous proxy (before the barrier that precedes the
// store).
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// The box at (c0, c1) (c0 innermost) of a 2-D tensor map from shared memory.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int c0,
                                             int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
            (unsigned long long)(uintptr_t)map),
        "r"(c0), "r"(c1), "r"(smem_addr(src))
        : "memory");
}

// Commit the stores issued so far and wait until they are complete (the
// hardware wait of the bulk-copy group: it ends when the copies have been
// written, not a spin loop).
__device__ __forceinline__ void tma_store_drain() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ------------------------------------------------------- transform tables
// Constants of the build (Taylor series in FP64, rounded once), the same for
// every handle.  w: for a radix-16 stage after Ns points (Ns = 2 .. 256) and
// k < Ns, the twiddles W^bk, W = exp(-2 pi i / 16 Ns), b = 2, 4, 6, 8, 1, 3,
// 12 at [8 (Ns - 2 + k)]; the others are one product of two of them (loads
// cost more than the multiplies).  A radix-8 stage's W, W^2, W^3 and W^4 are
// the first four (two 16-byte loads).  ph: exp(-i pi u / 2n) for u < n at
// [n - 16 + u].  Fewer loads and more products (W, W^2, W^4, W^8 only; ph
// from one load and constants) saved 1 to 2 % of the passes and raised the
// relative error of psi, E_x and E_y from 2.1-2.9 to 2.8-3.2 1e-7 at n = 2048
// and 4096 (shared-memory form: 2.3-3.0).
constexpr double kPi = 3.14159265358979323846;

struct UnitD {
    double c, s;
};

// sine and cosine series on [-pi/4, pi/4] (terms to a^23)
constexpr UnitD unit_small(double a) {
    double c = 1.0, s = a, tc = 1.0, ts = a;
    for (int k = 1; k < 12; ++k) {
        tc *= -a * a / ((2 * k - 1) * (2 * k));
        ts *= -a * a / ((2 * k) * (2 * k + 1));
        c += tc;
        s += ts;
    }
    return {c, s};
}

// cos and sin of 2 pi num / den (num >= 0)
constexpr UnitD unit_root(long num, long den) {
    num %= den;
    const long quad = (4 * num + den / 2) / den;   // nearest multiple of pi/2
    const UnitD u = unit_small(0.5 * kPi * (double)(4 * num - quad * den) / (double)den);
    switch (quad & 3) {
        case 0: return {u.c, u.s};
        case 1: return {-u.s, u.c};
        case 2: return {-u.c, -u.s};
        default: return {u.s, -u.c};
    }
}

struct Pair {
    float x, y;
};

constexpr int kMaxNs = FFTPL_MAX_N / 16;

struct alignas(16) SpecTables {
    Pair w[8 * (2 * kMaxNs - 2)];
    Pair ph[2 * FFTPL_MAX_N - 16];
};

constexpr SpecTables make_tables() {
    SpecTables t{};
    for (int ns = 2; ns <= kMaxNs; ns *= 2)
        for (int k = 0; k < ns; ++k)
            for (int b = 0; b < 7; ++b) {
                const int e[7] = {2, 4, 6, 8, 1, 3, 12};
                const UnitD u = unit_root((long)k * e[b], 16L * ns);
                t.w[8 * (ns - 2 + k) + b] = {(float)u.c, (float)-u.s};
            }
    for (int n = 16; n <= FFTPL_MAX_N; n *= 2)
        for (int k = 0; k < n; ++k) {
            const UnitD u = unit_root(k, 4L * n);
            t.ph[n - 16 + k] = {(float)u.c, (float)-u.s};
        }
    return t;
}

static __device__ const SpecTables g_tab = make_tables();

// exp(-i pi u / 2N)
template <int N>
__device__ __forceinline__ float2 phase(int u) {
    return __ldg(reinterpret_cast<const float2*>(g_tab.ph) + (N - 16 + u));
}

// ------------------------------------------------------------ FFT core
// Twiddle exp(-+2 pi i k / 16) for the small exponents a radix-16 butterfly
// uses (cos and sin of multiples of pi/8).
__device__ __forceinline__ float2 w16(int e, bool inv) {
    const float c1 = 0.92387953251128674f, s1 = 0.38268343236508978f, h = 0.70710678118654752f;
    float2 w;
    switch (e & 15) {
        case 0: w = make_float2(1.0f, 0.0f); break;
        case 1: w = make_float2(c1, -s1); break;
        case 2: w = make_float2(h, -h); break;
        case 3: w = make_float2(s1, -c1); break;
        case 4: w = make_float2(0.0f, -1.0f); break;
        case 6: w = make_float2(-h, -h); break;
        case 9: w = make_float2(-c1, s1); break;
        default: w = make_float2(1.0f, 0.0f); break;  // not used
    }
    if (inv) w.y = -w.y;
    return w;
}

// multiply by -i (forward) or +i (inverse)
__device__ __forceinline__ float2 rot(float2 a, bool inv) {
    return inv ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

__device__ __forceinline__ void dft2(float2& a, float2& b) {
    float2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}

// in-place 4-point DFT of (a0, a1, a2, a3)
__device__ __forceinline__ void dft4(float2& a0, float2& a1, float2& a2, float2& a3, bool inv) {
    float2 s02 = cadd(a0, a2), d02 = csub(a0, a2);
    float2 s13 = cadd(a1, a3), d13 = rot(csub(a1, a3), inv);
    a0 = cadd(s02, s13);
    a2 = csub(s02, s13);
    a1 = cadd(d02, d13);
    a3 = csub(d02, d13);
}

// 8-point DFT of v[0], v[S], .., v[7 S] in place, natural order
template <int S>
__device__ __forceinline__ void dft8(float2* v, bool inv) {
    // 8 = 2 x 4: DFT4 of even and odd samples, twiddle W8^k, combine
    float2 e0 = v[0], e1 = v[2 * S], e2 = v[4 * S], e3 = v[6 * S];
    float2 o0 = v[S], o1 = v[3 * S], o2 = v[5 * S], o3 = v[7 * S];
    dft4(e0, e1, e2, e3, inv);
    dft4(o0, o1, o2, o3, inv);
    o1 = cmul(o1, w16(2, inv));
    o2 = cmul(o2, w16(4, inv));
    o3 = cmul(o3, w16(6, inv));
    v[0] = cadd(e0, o0); v[4 * S] = csub(e0, o0);
    v[S] = cadd(e1, o1); v[5 * S] = csub(e1, o1);
    v[2 * S] = cadd(e2, o2); v[6 * S] = csub(e2, o2);
    v[3 * S] = cadd(e3, o3); v[7 * S] = csub(e3, o3);
}

// 16-point DFT in place, natural order
__device__ __forceinline__ void dft16(float2* v, bool inv) {
    // 16 = 4 x 4: X[k1 + 4 k2] = sum_n2 W4^(n2 k2) W16^(n2 k1) sum_n1 x[4 n1 + n2] W4^(n1 k1)
    float2 y[4][4];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
        y[n2][0] = v[n2]; y[n2][1] = v[n2 + 4]; y[n2][2] = v[n2 + 8]; y[n2][3] = v[n2 + 12];
        dft4(y[n2][0], y[n2][1], y[n2][2], y[n2][3], inv);
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1)
            if (n2 > 0) y[n2][k1] = cmul(y[n2][k1], w16(n2 * k1, inv));
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        float2 a0 = y[0][k1], a1 = y[1][k1], a2 = y[2][k1], a3 = y[3][k1];
        dft4(a0, a1, a2, a3, inv);
        v[k1] = a0; v[k1 + 4] = a1; v[k1 + 8] = a2; v[k1 + 12] = a3;
    }
}

// Elements per thread: 8 up to n = 1024, where a pass has fewer warps than
// the GPU has room for and the length of a thread's own chain decides, 16
// above, where fewer exchanges win.  A graph-replayed evaluation without nets
// (two memsets, scatter, the passes, cell kernel) of 1,000 cells, E = 8
// against E = 16: n = 64 17.8 / 22.5 us, 512 20.6 / 26.1, 1024 28.8 / 30.4,
// 2048 82.1 / 65.7, 4096 284 / 231.
constexpr int spec_elems(int logn) { return logn <= 10 ? 8 : 16; }
// Blocks of t threads per SM the registers are budgeted for: 16 warps of up
// to 128, or 24 of up to 80.
constexpr int spec_blocks(int logn, int t) {
    const int b = (spec_elems(logn) == 16 ? 512 : 768) / t;
    return b > 32 ? 32 : b;
}

// Layout of a pass: NF FFTs of length n side by side per group of
// NF n / E threads (FFT f = thread % NF, so that shared memory holds the NF
// elements of one index together), as many groups as fill a warp per block.
template <int LOGN, int NF>
struct Lay {
    static constexpr int N = 1 << LOGN;
    static constexpr int E = spec_elems(LOGN);   // elements per thread
    static constexpr int LOGE = E == 16 ? 4 : 3;
    static constexpr int Q = N / E;              // threads per FFT
    static constexpr int LT = NF * Q;            // threads per group
    static constexpr int GB = LT >= 32 ? 1 : 32 / LT;   // groups per block
    static constexpr int T = LT >= 32 ? LT : 32;        // threads per block
    static constexpr int R0 = 1 << (LOGN % LOGE);   // radix of the first stage (1: E)
    static constexpr int LQ = NF == 1 ? 4 : 3;      // log2(16 / NF)
    // elements of one padded buffer
    static constexpr int PADN = N + (R0 == 1 || (N >> LQ) < N / E ? N / E : (N >> LQ));
    // shared bytes of one group holding V buffers per FFT (128-byte multiple)
    static constexpr int group_bytes(int v) { return (v * NF * PADN * 8 + 127) / 128 * 128; }
};

// Thread's element offset t (elements t + Q q) such that thread Q - 1 - t of
// the same FFT is lane *partner of the same warp.
template <int LOGN, int NF>
__device__ __forceinline__ int lane_rev(int lt, int* partner) {
    using L = Lay<LOGN, NF>;
    const int lane = threadIdx.x & 31;
    if constexpr (L::LT <= 32) {
        const int t = lt / NF;
        *partner = lane + (L::Q - 1 - 2 * t) * NF;
        return t;
    } else {
        constexpr int half = 16 / NF;
        const int i = (lt >> 5) * half + (lane & 15) / NF;
        *partner = lane ^ 16;
        return lane < 16 ? i : L::Q - 1 - i;
    }
}

// The same with thread (Q - t) mod Q as the partner.
template <int LOGN, int NF>
__device__ __forceinline__ int lane_neg(int lt, int* partner) {
    using L = Lay<LOGN, NF>;
    const int lane = threadIdx.x & 31;
    if constexpr (L::LT <= 32) {
        const int t = lt / NF;
        *partner = lane + (((L::Q - t) & (L::Q - 1)) - t) * NF;
        return t;
    } else {
        constexpr int half = 16 / NF;
        const int i = (lt >> 5) * half + (lane & 15) / NF;
        *partner = i == 0 ? lane : lane ^ 16;
        return lane < 16 ? i : (i == 0 ? L::Q / 2 : L::Q - i);
    }
}

// Padding of the exchange after a stage, so that its strided writes spread
// over the banks: after the first small radix, and after a radix-E stage that
// followed Ns points.
template <int LQ>
__device__ __forceinline__ int pad_first(int i) { return i + (i >> LQ); }
template <int E, int Ns>
__device__ __forceinline__ int pad_stage(int i) {
    if constexpr (Ns < 16) return i + Ns * (i / (E * Ns));
    else return i;
}

template <int LOGN, int NF>
__device__ __forceinline__ void group_sync() {
    if constexpr (Lay<LOGN, NF>::T == 32) __syncwarp();
    else __syncthreads();
}

__device__ __forceinline__ float2 shfl2(float2 v, int src) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// Twiddles W^r, r < E, of a radix-E stage from the table's entry.
template <int E>
struct Tw {
    float4 a, b, c;
    float2 d;
    __device__ __forceinline__ void load(int Ns, int k) {
        const float4* tb = reinterpret_cast<const float4*>(g_tab.w) + 4 * (Ns - 2 + k);
        a = __ldg(tb);
        b = __ldg(tb + 1);
        if (E == 16) {
            c = __ldg(tb + 2);
            d = __ldg(reinterpret_cast<const float2*>(tb + 3));
        }
    }
    template <int NV>
    __device__ __forceinline__ void apply(float2 (&v)[NV][E], bool inv) const {
        const float s = inv ? -1.0f : 1.0f;
        float2 w[E];
        if constexpr (E == 16) {
            w[2] = make_float2(a.x, s * a.y);
            w[4] = make_float2(a.z, s * a.w);
            w[6] = make_float2(b.x, s * b.y);
            w[8] = make_float2(b.z, s * b.w);
            w[1] = make_float2(c.x, s * c.y);
            w[3] = make_float2(c.z, s * c.w);
            w[12] = make_float2(d.x, s * d.y);
            w[5] = cmul(w[4], w[1]);
            w[7] = cmul(w[4], w[3]);
            w[9] = cmul(w[8], w[1]);
            w[10] = cmul(w[8], w[2]);
            w[11] = cmul(w[8], w[3]);
            w[13] = cmul(w[12], w[1]);
            w[14] = cmul(w[12], w[2]);
            w[15] = cmul(w[12], w[3]);
        } else {
            w[1] = make_float2(a.x, s * a.y);
            w[2] = make_float2(a.z, s * a.w);
            w[3] = make_float2(b.x, s * b.y);
            w[4] = make_float2(b.z, s * b.w);
            w[5] = cmul(w[4], w[1]);
            w[6] = cmul(w[4], w[2]);
            w[7] = cmul(w[4], w[3]);
        }
#pragma unroll
        for (int i = 0; i < NV; ++i)
#pragma unroll
            for (int r = 1; r < E; ++r) v[i][r] = cmul(v[i][r], w[r]);
    }
};

template <int E>
__device__ __forceinline__ void dft_full(float2* v, bool inv) {
    if constexpr (E == 16) dft16(v, inv);
    else dft8<1>(v, inv);
}

// The radix-E stages from Ns points on; the elements of index i of FFT f are
// in buf[PAD(i) NF + f] (PNs > 0: padded by a radix-E stage after PNs points,
// 0: by the first small radix).
template <int LOGN, int NF, int NV, int Ns, int PNs, int E>
__device__ __forceinline__ void fft_stages(float2 (&v)[NV][E], float2* buf, int lt, int tl, int f,
                                           bool inv) {
    using L = Lay<LOGN, NF>;
    if constexpr (Ns < L::N) {
        constexpr bool last = E * Ns == L::N;
        const int t = last ? tl : lt / NF;
        const int k = t & (Ns - 1);
        Tw<E> tw;
        tw.load(Ns, k);
        group_sync<LOGN, NF>();
#pragma unroll
        for (int a = 0; a < NV; ++a)
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int i = t + L::Q * q;
                const int p = PNs == 0 ? pad_first<L::LQ>(i) : pad_stage<E, (PNs ? PNs : 1)>(i);
                v[a][q] = buf[a * (NF * L::PADN) + p * NF + f];
            }
        tw.apply(v, inv);
#pragma unroll
        for (int a = 0; a < NV; ++a) dft_full<E>(v[a], inv);
        if constexpr (!last) {
            group_sync<LOGN, NF>();
            const int o = (t - k) * E + k;
#pragma unroll
            for (int a = 0; a < NV; ++a)
#pragma unroll
                for (int r = 0; r < E; ++r)
                    buf[a * (NF * L::PADN) + pad_stage<E, Ns>(o + r * Ns) * NF + f] = v[a][r];
            fft_stages<LOGN, NF, NV, E * Ns, Ns>(v, buf, lt, tl, f, inv);
        }
    }
}

// NV complex FFTs of length N per thread group and f: thread element offset
// t0 on input, tl on output (elements t + Q q in natural order).  Forward:
// X[k] = sum x[j] exp(-2 pi i jk / N); inverse: + sign, no 1/N.  buf (NV
// buffers of NF PADN elements) must be free on entry; the caller
// synchronises before it uses buf again.
template <int LOGN, int NF, int NV, int E>
__device__ __forceinline__ void fft_regs(float2 (&v)[NV][E], float2* buf, int lt, int t0, int tl,
                                         int f, bool inv) {
    using L = Lay<LOGN, NF>;
    constexpr int R0 = L::R0;
    if constexpr (R0 == 1) {
#pragma unroll
        for (int a = 0; a < NV; ++a) dft_full<E>(v[a], inv);
        if constexpr (L::N > E) {
#pragma unroll
            for (int a = 0; a < NV; ++a)
#pragma unroll
                for (int r = 0; r < E; ++r)
                    buf[a * (NF * L::PADN) + pad_stage<E, 1>(E * t0 + r) * NF + f] = v[a][r];
            fft_stages<LOGN, NF, NV, E, 1>(v, buf, lt, tl, f, inv);
        }
    } else {
        constexpr int C = E / R0;   // butterflies per thread: j = t0 + Q i, inputs v[i + C r]
#pragma unroll
        for (int a = 0; a < NV; ++a) {
#pragma unroll
            for (int i = 0; i < C; ++i) {
                float2* x = v[a] + i;
                if constexpr (R0 == 2) dft2(x[0], x[C]);
                else if constexpr (R0 == 4) dft4(x[0], x[C], x[2 * C], x[3 * C], inv);
                else dft8<C>(x, inv);
            }
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int o = (t0 + L::Q * (q % C)) * R0 + q / C;
                buf[a * (NF * L::PADN) + pad_first<L::LQ>(o) * NF + f] = v[a][q];
            }
        }
        fft_stages<LOGN, NF, NV, R0, 0>(v, buf, lt, tl, f, inv);
    }
}

// The two real spectra of a packed pair at u, from Z[u] and Z[n-u], times 2:
// V_1 = Z[u] + conj Z[n-u], V_2 = (Z[u] - conj Z[n-u]) / i.
__device__ __forceinline__ void split_pair(float2 zu, float2 zn, float2* v1, float2* v2) {
    *v1 = make_float2(zu.x + zn.x, zu.y - zn.y);
    *v2 = make_float2(zu.y + zn.y, zn.x - zu.x);
}

// Spectrum of an inverse-cosine pair packed for one complex IFFT.  For the
// sums y1 = sum c1[u] C(u,.), y2 = sum c2[u] C(u,.), with ct[0] = c[0],
// ct[u] = c[u]/2 (u >= 1), ct[N] = 0:
//   Z[u] = exp(i pi u / 2N) * ((ct1[u] + ct2[N-u]) + i (ct2[u] - ct1[N-u]))
// and then y1 + i y2 = unshuffle(IFFT(Z)).
__device__ __forceinline__ float2 pack_inv(float c1u, float c1nu, float c2u, float c2nu, float2 ph) {
    float re = c1u + c2nu, im = c2u - c1nu;
    // multiply by conj(ph) = exp(+i pi u / 2N)
    return make_float2(re * ph.x + im * ph.y, im * ph.x - re * ph.y);
}

// Sample of the natural order held at position k of the reordering.
__device__ __forceinline__ int mk_src(int y, int N) { return (y & 1) ? (N - 1 - (y >> 1)) : (y >> 1); }

// A group's finished tile [N/2][8 floats] to columns c0 .. c0+7 of a
// transposed map of N/2 rows of 2N floats: one thread through the TMA unit,
// or every thread of the group with plain stores.
template <int LOGN>
__device__ __forceinline__ void store_tile(const float4* tile, float* dst, const CUtensorMap* map,
                                           int c0, int lt, int nthreads, bool tma) {
    constexpr int N = 1 << LOGN, ROWS = N / 2, BOX = ROWS < 256 ? ROWS : 256;
    if (tma) {
        if (lt == 0)
            for (int b = 0; b < ROWS / BOX; ++b) tma_store_2d(map, tile + 2 * b * BOX, c0, b * BOX);
    } else {
        for (int i = lt; i < 2 * ROWS; i += nthreads)
            *reinterpret_cast<float4*>(dst + (size_t)(i >> 1) * (2 * N) + c0 + 4 * (i & 1)) = tile[i];
    }
}

// -------------------------------------------------------- pass 1: rows
// Group: 4 rows y0 .. y0+3 of rho (2 per complex FFT) -> T1[u/2][y0..y0+3].
template <int LOGN, bool QUANT>
__global__ void __launch_bounds__(Lay<LOGN, 2>::T, spec_blocks(LOGN, Lay<LOGN, 2>::T))
k_rows_fwd(const float* D, const long long* Dq,
           const float* __restrict__ M, float inv_ab, float cap, float* __restrict__ T1,
           double* __restrict__ acc, DetRed dr, const __grid_constant__ CUtensorMap mT1, int tma) {
    using L = Lay<LOGN, 2>;
    constexpr int N = L::N, Q = L::Q, E = L::E;
    extern __shared__ __align__(128) unsigned char smem[];
    const int g = L::GB == 1 ? 0 : threadIdx.x / L::LT;
    const int lt = L::GB == 1 ? threadIdx.x : threadIdx.x % L::LT;
    const int gi = blockIdx.x * L::GB + g, f = lt & 1;
    const bool live = gi < N / 4;
    const int y0 = 4 * (live ? gi : N / 4 - 1);
    float2* buf = reinterpret_cast<float2*>(smem + g * L::group_bytes(1));
    if (smem_addr(smem) & 127u) tma = 0;   // the TMA unit's source alignment
    int pa, pb;
    const int ta = lane_rev<LOGN, 2>(lt, &pa);
    chain_wait();
    chain_trigger();
    // per-thread sums of 2 E non-negative terms in float32
    float tau = 0.0f, charge = 0.0f;
    float2 v[1][E];
    // all of D's loads first
    const size_t b = (size_t)(y0 + 2 * f) * N + 2 * ta;
    typename std::conditional<QUANT, longlong2, float2>::type dd[2][E / 2];
#pragma unroll
    for (int q = 0; q < E / 2; ++q) {
        const size_t b0 = b + 2 * Q * q;
        if constexpr (QUANT) {
            dd[0][q] = ld_dep(reinterpret_cast<const longlong2*>(Dq + b0));
            dd[1][q] = ld_dep(reinterpret_cast<const longlong2*>(Dq + b0 + N));
        } else {
            dd[0][q] = ld_dep(reinterpret_cast<const float2*>(D + b0));
            dd[1][q] = ld_dep(reinterpret_cast<const float2*>(D + b0 + N));
        }
    }
#pragma unroll
    for (int q = 0; q < E / 2; ++q) {
        // samples 2p and 2p+1 of both rows, p = ta + Q q: elements p and N-1-p
        const size_t b0 = b + 2 * Q * q, b1 = b0 + N;
        float d[4], mm[4];
        const float2 m0 = __ldg(reinterpret_cast<const float2*>(M + b0));
        const float2 m1 = __ldg(reinterpret_cast<const float2*>(M + b1));
        mm[0] = m0.x; mm[1] = m0.y; mm[2] = m1.x; mm[3] = m1.y;
        d[0] = (float)dd[0][q].x; d[1] = (float)dd[0][q].y;
        d[2] = (float)dd[1][q].x; d[3] = (float)dd[1][q].y;
        if (QUANT)
            for (int t = 0; t < 4; ++t) d[t] *= 2.3283064365386963e-10f;
        float rv[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            tau += fmaxf(0.0f, d[t] - (cap - mm[t]));
            charge += d[t] + mm[t];
            rv[t] = (d[t] + mm[t]) * inv_ab;
        }
        v[0][q] = make_float2(rv[0], rv[2]);
        v[0][E - 1 - q] = shfl2(make_float2(rv[1], rv[3]), pa);
    }
    const int k = lane_neg<LOGN, 2>(lt, &pb);
    fft_regs<LOGN, 2, 1>(v, buf, lt, ta, k, f, false);
    group_sync<LOGN, 2>();   // the tile replaces the exchange buffer
    // split the packed spectra and apply the post-twiddle: A_j[u] = Re(ph[u] V_j[u])
    float* tile = reinterpret_cast<float*>(buf);
#pragma unroll
    for (int r = 0; r < E; ++r) {
        float2 zn = shfl2(v[0][E - 1 - r], pb), v1, v2;
        if (k == 0) zn = v[0][(E - r) & (E - 1)];
        split_pair(v[0][r], zn, &v1, &v2);
        const float2 p = phase<N>(k + Q * r);
        const int u = k + Q * r;
        float* dst = tile + (u >> 1) * 8 + 4 * f + (u & 1);
        dst[0] = 0.5f * (v1.x * p.x - v1.y * p.y);
        dst[2] = 0.5f * (v2.x * p.x - v2.y * p.y);
    }
    if (tma) fence_async_smem();
    group_sync<LOGN, 2>();
    if (live) store_tile<LOGN>(reinterpret_cast<const float4*>(tile), T1, &mT1, 2 * y0, lt, L::LT, tma);
    reduce2(live ? tau : 0.0f, live ? charge : 0.0f, acc, ACC_TAU, ACC_CHARGE, dr);
    if (tma && live && lt == 0) tma_store_drain();
}

// ------------------------------------------------- pass 2: columns
// One spectral element of two rows (u, u+1) at v: from Z[v] and Z[n-v] the
// DCT-II values, the divide, the energy terms and the packed inputs of the
// inverse sums P (cosine sum of Psi) and R (sine sum of w_v Psi as a cosine
// sum of c2[v'] = s[N-v'], s[v] = w_v Psi[v], c2[0] = 0).
struct SpecRow {
    float w2a, w2b;   // w_u^2 + eps of the two rows
    float ha, hb;     // eps_u / 2n^2
    bool drop;        // row u = 0 without the Helmholtz term: the (0,0) mode dropped
};

__device__ __forceinline__ void spectral_elem(float2 zu, float2 zn, float2 p, float wv, float wn,
                                              bool v0, const SpecRow& s, float2* zp, float2* zr,
                                              dfloat* energy) {
    float2 v1, v2;
    split_pair(zu, zn, &v1, &v2);
    // ph[n-v] = -i conj(ph[v]): both values of a pair from one product
    const float2 wa = cmul(p, v1), wb = cmul(p, v2);
    const float ba = wa.x, bna = -wa.y, bb = wb.x, bnb = -wb.y;   // twice B
    // the divisors are at least (pi/L)^2 > 0 (or eps): the fast divide (2 ulp)
    // stays far inside the transform's bound
    const float wv2 = wv * wv, wn2 = wn * wn;
    float ca = __fdividef(s.ha * ba, wv2 + s.w2a);
    const float cb = __fdividef(s.hb * bb, wv2 + s.w2b);
    float na = __fdividef(s.ha * bna, wn2 + s.w2a);
    float nb = __fdividef(s.hb * bnb, wn2 + s.w2b);
    if (v0) {
        if (s.drop) ca = 0.0f;   // Poisson: no (0,0) mode
        na = 0.0f;
        nb = 0.0f;
    }
    // B Psi: Psi = 2 ct but at v = 0 (ct = Psi); B is half of ba
    const float ea = ba * ca, eb = bb * cb;
    sum2_add(*energy, v0 ? 0.5f * ea : ea);
    sum2_add(*energy, v0 ? 0.5f * eb : eb);
    *zp = pack_inv(ca, na, cb, nb, p);
    *zr = pack_inv(wn * na, wv * ca, wn * nb, wv * cb, p);
}

// Group: 4 rows u0 .. u0+3 of T1.  Forward DCT-II along y, spectral divide,
// energy, then the inverse sums along y.  Each complex IFFT carries the same
// quantity for two rows (P with P, R with R), so both parts share a scale.
// The forward FFT ends in each thread with the elements its inverse FFTs
// begin with, so the spectrum never leaves the registers.
template <int LOGN>
__global__ void __launch_bounds__(Lay<LOGN, 2>::T, spec_blocks(LOGN, Lay<LOGN, 2>::T))
k_cols(const float* T1, float* __restrict__ PT, float* __restrict__ RT, float pi_lx,
       float pi_ly, float eps, double* __restrict__ acc, DetRed dr,
       const __grid_constant__ CUtensorMap mPT, const __grid_constant__ CUtensorMap mRT, int tma) {
    using L = Lay<LOGN, 2>;
    constexpr int N = L::N, Q = L::Q, E = L::E;
    extern __shared__ __align__(128) unsigned char smem[];
    const int g = L::GB == 1 ? 0 : threadIdx.x / L::LT;
    const int lt = L::GB == 1 ? threadIdx.x : threadIdx.x % L::LT;
    const int gi = blockIdx.x * L::GB + g, f = lt & 1;
    const bool live = gi < N / 4;
    const int u0 = 4 * (live ? gi : N / 4 - 1);
    float2* buf = reinterpret_cast<float2*>(smem + g * L::group_bytes(2));
    if (smem_addr(smem) & 127u) tma = 0;
    int pa, pb;
    const int ta = lane_rev<LOGN, 2>(lt, &pa);
    float2 z[2][E];
    dfloat energy = df_zero();
    int k;
    {
        float2 v[1][E];
        chain_wait();
        chain_trigger();
        const float4* row = reinterpret_cast<const float4*>(T1 + (size_t)(u0 / 2 + f) * (2 * N));
#pragma unroll
        for (int q = 0; q < E / 2; ++q) {
            const float4 a = ld_dep(row + ta + Q * q);   // samples 2p, 2p+1 of both rows
            v[0][q] = make_float2(a.x, a.y);
            v[0][E - 1 - q] = make_float2(a.z, a.w);
        }
#pragma unroll
        for (int q = E / 2; q < E; ++q) v[0][q] = shfl2(v[0][q], pa);
        k = lane_neg<LOGN, 2>(lt, &pb);
        fft_regs<LOGN, 2, 1>(v, buf, lt, ta, k, f, false);
        SpecRow s;
        const int u = u0 + 2 * f;
        const float wa = pi_lx * (float)u, wb = pi_lx * (float)(u + 1);
        const float invn2 = 1.0f / ((float)N * (float)N);
        s.w2a = fmaf(wa, wa, eps);
        s.w2b = fmaf(wb, wb, eps);
        s.ha = (u == 0 ? 0.5f : 1.0f) * invn2;
        s.hb = invn2;
        s.drop = u == 0 && !(eps > 0.0f);
        const float kf = (float)k;
        // pairs (r, E - 1 - r): each needs the other's element of the partner
        // (element E - r of the own thread at k = 0)
        float2 hi = v[0][0];
#pragma unroll
        for (int r = 0; r < E / 2; ++r) {
            const float2 a = v[0][r], b = v[0][E - 1 - r];
            float2 na = shfl2(b, pb), nb = shfl2(a, pb);
            if (k == 0) {
                na = hi;
                nb = v[0][r + 1];
            }
            hi = b;
            const float va = kf + (float)(Q * r), vb = kf + (float)(Q * (E - 1 - r));
            spectral_elem(a, na, phase<N>(k + Q * r), pi_ly * va, pi_ly * ((float)N - va),
                          r == 0 && k == 0, s, &z[0][r], &z[1][r], &energy);
            spectral_elem(b, nb, phase<N>(k + Q * (E - 1 - r)), pi_ly * vb, pi_ly * ((float)N - vb), false,
                          s, &z[0][E - 1 - r], &z[1][E - 1 - r], &energy);
        }
    }
    group_sync<LOGN, 2>();   // the forward exchange has been read
    fft_regs<LOGN, 2, 2>(z, buf, lt, k, ta, f, true);
    group_sync<LOGN, 2>();   // the tiles replace the exchange buffers
    // unshuffle: y = 2o <- element o, y = 2o+1 <- element N-1-o; R times (-1)^y
    float4* tP = reinterpret_cast<float4*>(buf);
    float4* tR = tP + N;
#pragma unroll
    for (int q = 0; q < E / 2; ++q) {
        const int o = ta + Q * q;
        const float2 p0 = z[0][q], p1 = shfl2(z[0][E - 1 - q], pa);
        const float2 r0 = z[1][q], r1 = shfl2(z[1][E - 1 - q], pa);
        tP[2 * o + f] = make_float4(p0.x, p1.x, p0.y, p1.y);
        tR[2 * o + f] = make_float4(r0.x, -r1.x, r0.y, -r1.y);
    }
    if (tma) fence_async_smem();
    group_sync<LOGN, 2>();
    if (live) {
        store_tile<LOGN>(tP, PT, &mPT, 2 * u0, lt, L::LT, tma);
        store_tile<LOGN>(tR, RT, &mRT, 2 * u0, lt, L::LT, tma);
    }
    reduce2(live ? df_val(energy) : 0.0f, 0.0f, acc, ACC_N, -1, dr);
    if (tma && live && lt == 0) tma_store_drain();
}

// ------------------------------------------------- pass 3: inverse rows
// Coefficients c[t + Q q] of two rows (re, im) and their partners, packed in
// place for the inverse FFT: the cosine sum of c (SINE = false), or the
// reversed coefficients w_u c of the sine sum (c'[u] = w_{N-u} c[N-u],
// c'[0] = 0), whose cosine sum times (-1)^x is the sine sum.
template <int LOGN, bool SINE>
__device__ __forceinline__ void pack_rows(const float2 (&c)[spec_elems(LOGN)], float2* z, int k,
                                          int pb, float pi_lx) {
    constexpr int N = 1 << LOGN, E = spec_elems(LOGN), Q = N / E;
    const float kf = (float)k;
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const float2 a = c[r];
        float2 n = shfl2(c[E - 1 - r], pb);
        if (k == 0) n = r == 0 ? make_float2(0.0f, 0.0f) : c[(E - r) & (E - 1)];
        const float2 p = phase<N>(k + Q * r);
        if (SINE) {
            const float u = kf + (float)(Q * r);
            const float wu = 0.5f * (pi_lx * u), wn = 0.5f * (pi_lx * ((float)N - u));
            // u = 0: both coefficients vanish (n = 0 and w_0 = 0)
            z[r] = pack_inv(wn * n.x, wu * a.x, wn * n.y, wu * a.y, p);
        } else {
            const float h = r == 0 && k == 0 ? 1.0f : 0.5f;   // c[0] is not halved
            z[r] = pack_inv(h * a.x, 0.5f * n.x, h * a.y, 0.5f * n.y, p);
        }
    }
}

// What an inverse-row pass writes: the interleaved field of the evaluation,
// the potential alone (on demand), or the three separate maps of a solve.
enum { INV_FIELD, INV_PSI, INV_MAPS };

// Group: one pair of rows y, y+1.  E_x (the sine sum of w_u P) and E_y (the
// cosine sum of R) in one round of two inverse FFTs; psi (the cosine sum of
// P) is not needed by the evaluation (the energy comes from the column pass
// by Parseval).
template <int LOGN, int WHAT>
__global__ void __launch_bounds__(Lay<LOGN, 1>::T, spec_blocks(LOGN, Lay<LOGN, 1>::T))
k_rows_inv(const float* PT, const float* RT, float2* __restrict__ E2,
           float* __restrict__ psi, float* __restrict__ ex, float* __restrict__ ey, float pi_lx) {
    using L = Lay<LOGN, 1>;
    constexpr int N = L::N, Q = L::Q, E = L::E;
    extern __shared__ __align__(128) unsigned char smem[];
    const int g = L::GB == 1 ? 0 : threadIdx.x / L::LT;
    const int lt = L::GB == 1 ? threadIdx.x : threadIdx.x % L::LT;
    const int gi = blockIdx.x * L::GB + g;
    const bool live = gi < N / 2;
    const int j = live ? gi : N / 2 - 1;
    constexpr int NV = WHAT == INV_PSI ? 1 : 2;
    float2* buf = reinterpret_cast<float2*>(smem + g * L::group_bytes(NV));
    int pa, pb;
    const int ta = lane_rev<LOGN, 1>(lt, &pa), k = lane_neg<LOGN, 1>(lt, &pb);
    const float2* pr = reinterpret_cast<const float2*>(PT) + (size_t)j * N + k;
    const float2* rr = reinterpret_cast<const float2*>(RT) + (size_t)j * N + k;
    const size_t row0 = (size_t)(2 * j) * N, row1 = row0 + N;
    chain_wait();
    chain_trigger();
    if (WHAT != INV_PSI) {
        float2 z[2][E];
        {
            float2 c[E], e[E];
#pragma unroll
            for (int q = 0; q < E; ++q) {
                c[q] = ld_dep(pr + Q * q);
                e[q] = ld_dep(rr + Q * q);
            }
            pack_rows<LOGN, true>(c, z[0], k, pb, pi_lx);
            pack_rows<LOGN, false>(e, z[1], k, pb, pi_lx);
        }
        fft_regs<LOGN, 1, 2>(z, buf, lt, k, ta, 0, true);
#pragma unroll
        for (int q = 0; q < E / 2; ++q) {
            const int o = ta + Q * q;   // samples 2o, 2o+1 of both rows
            const float2 x0 = z[0][q], x1 = shfl2(z[0][E - 1 - q], pa);
            const float2 e0 = z[1][q], e1 = shfl2(z[1][E - 1 - q], pa);
            if (!live) continue;
            if (WHAT == INV_FIELD) {
                reinterpret_cast<float4*>(E2 + row0)[o] = make_float4(x0.x, e0.x, -x1.x, e1.x);
                reinterpret_cast<float4*>(E2 + row1)[o] = make_float4(x0.y, e0.y, -x1.y, e1.y);
            } else {
                reinterpret_cast<float2*>(ex + row0)[o] = make_float2(x0.x, -x1.x);
                reinterpret_cast<float2*>(ex + row1)[o] = make_float2(x0.y, -x1.y);
                reinterpret_cast<float2*>(ey + row0)[o] = make_float2(e0.x, e1.x);
                reinterpret_cast<float2*>(ey + row1)[o] = make_float2(e0.y, e1.y);
            }
        }
    }
    if (WHAT != INV_FIELD) {
        float2 z[1][E];
        {
            float2 c[E];
#pragma unroll
            for (int q = 0; q < E; ++q) c[q] = ld_dep(pr + Q * q);
            pack_rows<LOGN, false>(c, z[0], k, pb, pi_lx);
        }
        if (WHAT == INV_MAPS) group_sync<LOGN, 1>();   // the field's exchange has been read
        fft_regs<LOGN, 1, 1>(z, buf, lt, k, ta, 0, true);
#pragma unroll
        for (int q = 0; q < E / 2; ++q) {
            const int o = ta + Q * q;
            const float2 s0 = z[0][q], s1 = shfl2(z[0][E - 1 - q], pa);
            if (!live) continue;
            reinterpret_cast<float2*>(psi + row0)[o] = make_float2(s0.x, s1.x);
            reinterpret_cast<float2*>(psi + row1)[o] = make_float2(s0.y, s1.y);
        }
    }
}

// ------------------------------------- tensor-core radix path: the rows
// The solve path FFTPL_SOLVE_TC_RADIX (k_tc.cu) computes every complex DFT
// of length n as two small dense products on the tensor cores.  These
// kernels do the same pre- and post-processing as the three passes above,
// row by row in global memory: Z holds complex rows of length n (Makhoul's
// packing of two real rows, or the packed spectrum of an inverse pair) that
// go into the DFT, V the complex rows that come out.

// rho rows (2r, 2r+1) packed: Z[r][k] = rho_2r[2k] + i rho_2r+1[2k] (k < n/2),
// Z[r][n-1-k] = rho_2r[2k+1] + i rho_2r+1[2k+1]; with the overflow and charge
// sums of k_rows_fwd.
template <bool QUANT>
__global__ void __launch_bounds__(256)
k_tcr_pack_rho(int n, int rows2, const float* __restrict__ D, const long long* __restrict__ Dq,
               const float* __restrict__ M, float inv_ab, float cap, float2* __restrict__ Z,
               double* __restrict__ acc, DetRed dr) {
    const int half = n >> 1;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    float tau = 0.0f, charge = 0.0f;
    if (q < (long long)rows2 * half) {
        const int r = (int)(q / half), k = (int)(q % half);
        const size_t b0 = (size_t)(2 * r) * n + 2 * k, b1 = b0 + n;
        float d[4], mm[4];
        const float2 m0 = *reinterpret_cast<const float2*>(M + b0);
        const float2 m1 = *reinterpret_cast<const float2*>(M + b1);
        mm[0] = m0.x; mm[1] = m0.y; mm[2] = m1.x; mm[3] = m1.y;
        if (QUANT) {
            const longlong2 q0 = *reinterpret_cast<const longlong2*>(Dq + b0);
            const longlong2 q1 = *reinterpret_cast<const longlong2*>(Dq + b1);
            d[0] = (float)q0.x * 2.3283064365386963e-10f;
            d[1] = (float)q0.y * 2.3283064365386963e-10f;
            d[2] = (float)q1.x * 2.3283064365386963e-10f;
            d[3] = (float)q1.y * 2.3283064365386963e-10f;
        } else {
            const float2 v0 = *reinterpret_cast<const float2*>(D + b0);
            const float2 v1 = *reinterpret_cast<const float2*>(D + b1);
            d[0] = v0.x; d[1] = v0.y; d[2] = v1.x; d[3] = v1.y;
        }
        float rv[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            tau += fmaxf(0.0f, d[t] - (cap - mm[t]));
            charge += d[t] + mm[t];
            rv[t] = (d[t] + mm[t]) * inv_ab;
        }
        float2* zr = Z + (size_t)r * n;
        zr[k] = make_float2(rv[0], rv[2]);
        zr[n - 1 - k] = make_float2(rv[1], rv[3]);
    }
    reduce2(tau, charge, acc, ACC_TAU, ACC_CHARGE, dr);
}

// Rows (2r, 2r+1) of a real map packed the same way (no sums).
__global__ void __launch_bounds__(256)
k_tcr_pack_rows(int n, int rows2, const float* __restrict__ A, float2* __restrict__ Z) {
    const int half = n >> 1;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)rows2 * half) return;
    const int r = (int)(q / half), k = (int)(q % half);
    const size_t b0 = (size_t)(2 * r) * n + 2 * k;
    const float2 a = *reinterpret_cast<const float2*>(A + b0);
    const float2 c = *reinterpret_cast<const float2*>(A + b0 + n);
    float2* zr = Z + (size_t)r * n;
    zr[k] = make_float2(a.x, c.x);
    zr[n - 1 - k] = make_float2(a.y, c.y);
}

// DCT-II spectra of packed pairs: A_j[u] = Re(ph[u] V_j[u]) with
// V_1 = (Z[u] + conj Z[n-u]) / 2, V_2 = (Z[u] - conj Z[n-u]) / 2i, the two
// rows of pair r; written transposed, T[u][8 g .. 8 g + 7] for the 4 pairs
// of group g (as k_rows_fwd writes T1).
__global__ void __launch_bounds__(256)
k_tcr_post_fwd(int n, int groups, const float2* __restrict__ V, const float2* __restrict__ ph,
               float* __restrict__ T) {
    const int half = n / 2 + 1;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)groups * half) return;
    const int g = (int)(q / half), u = (int)(q % half);
    float a[8], an[8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float2* vr = V + (size_t)(4 * g + t) * n;
        const float2 zu = vr[u & (n - 1)], zn = vr[(n - u) & (n - 1)];
        const float2 v1 = make_float2(0.5f * (zu.x + zn.x), 0.5f * (zu.y - zn.y));
        const float2 v2 = make_float2(0.5f * (zu.y + zn.y), 0.5f * (zn.x - zu.x));
        const float2 p = ph[u], pn = ph[n - u];
        a[2 * t] = v1.x * p.x - v1.y * p.y;
        a[2 * t + 1] = v2.x * p.x - v2.y * p.y;
        an[2 * t] = v1.x * pn.x + v1.y * pn.y;
        an[2 * t + 1] = v2.x * pn.x + v2.y * pn.y;
    }
    float4* dst = reinterpret_cast<float4*>(T + (size_t)(u & (n - 1)) * n + 8 * g);
    dst[0] = make_float4(a[0], a[1], a[2], a[3]);
    dst[1] = make_float4(a[4], a[5], a[6], a[7]);
    if (u > 0 && u < n / 2) {
        float4* dn = reinterpret_cast<float4*>(T + (size_t)(n - u) * n + 8 * g);
        dn[0] = make_float4(an[0], an[1], an[2], an[3]);
        dn[1] = make_float4(an[4], an[5], an[6], an[7]);
    }
}

// Column spectra of u-row pairs r (V, as in k_cols): divide by
// w_u^2 + w_v^2 (+ eps), drop the (0,0) mode, the energy, and the packed
// inverse inputs: Z[r] for P (cosine sums of Psi), Z[rows2 + r] for R
// (cosine sums of the reversed w_v Psi).
__global__ void __launch_bounds__(256)
k_tcr_spectral(int n, int rows2, const float2* __restrict__ V, const float2* __restrict__ ph,
               float pi_lx, float pi_ly, float eps, float2* __restrict__ Z,
               double* __restrict__ acc, DetRed dr) {
    const int half = n / 2 + 1;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    dfloat energy = df_zero();
    if (q < (long long)rows2 * half) {
        const int r = (int)(q / half), v = (int)(q % half);
        const float2* vr = V + (size_t)r * n;
        const float2 zu = vr[v & (n - 1)], zn = vr[(n - v) & (n - 1)];
        const float2 v1 = make_float2(0.5f * (zu.x + zn.x), 0.5f * (zu.y - zn.y));
        const float2 v2 = make_float2(0.5f * (zu.y + zn.y), 0.5f * (zn.x - zu.x));
        const float2 p = ph[v], qq = ph[n - v];
        float B[2][2];
        B[0][0] = v1.x * p.x - v1.y * p.y;
        B[1][0] = v2.x * p.x - v2.y * p.y;
        B[0][1] = v1.x * qq.x + v1.y * qq.y;
        B[1][1] = v2.x * qq.x + v2.y * qq.y;
        const float invn2 = 1.0f / ((float)n * (float)n);
        const float wv = pi_ly * (float)v, wvn = pi_ly * (float)(n - v);
        const float ev = (v == 0) ? 1.0f : 2.0f;
        const bool has_n = (v > 0 && v < n / 2);
        float c1v[2], c1n[2], c2v[2], c2n[2];
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            const int u = 2 * r + rr;
            const float wu = pi_lx * (float)u;
            const float eu = (u == 0) ? 1.0f : 2.0f;
            const float a0 = eu * ev * invn2 * B[rr][0];
            const float psi0 = (u == 0 && v == 0 && !(eps > 0.0f))
                                   ? 0.0f
                                   : __fdividef(a0, wu * wu + wv * wv + eps);
            float psin = 0.0f;
            if (has_n) {
                const float an = eu * 2.0f * invn2 * B[rr][1];
                psin = __fdividef(an, wu * wu + wvn * wvn + eps);
                energy = df_add(energy, B[rr][1] * psin);
            }
            energy = df_add(energy, B[rr][0] * psi0);
            c1v[rr] = (v == 0) ? psi0 : 0.5f * psi0;
            c1n[rr] = 0.5f * psin;
            c2v[rr] = (v == 0) ? 0.0f : 0.5f * wvn * psin;
            c2n[rr] = (v == 0) ? 0.0f : 0.5f * wv * psi0;
            if (v == n / 2) {
                c1n[rr] = c1v[rr];
                c2v[rr] = 0.5f * wv * psi0;
                c2n[rr] = c2v[rr];
            }
        }
        float2* zp = Z + (size_t)r * n;
        float2* zr = Z + (size_t)(rows2 + r) * n;
        zp[v & (n - 1)] = pack_inv(c1v[0], c1n[0], c1v[1], c1n[1], p);
        zr[v & (n - 1)] = pack_inv(c2v[0], c2n[0], c2v[1], c2n[1], p);
        if (has_n) {
            zp[n - v] = pack_inv(c1n[0], c1v[0], c1n[1], c1v[1], qq);
            zr[n - v] = pack_inv(c2n[0], c2v[0], c2n[1], c2v[1], qq);
        }
    }
    reduce2(df_val(energy), 0.0f, acc, ACC_N, -1, dr);
}

// Inverse outputs of the column pass: pair r of P (V[r]) and of R
// (V[rows2 + r]) unshuffled (y = 2j <- position j, y = 2j+1 <- n-1-j; R times
// (-1)^y) and written transposed, PT[j][8 g .. 8 g + 7] (two rows y
// interleaved), RT likewise.
__global__ void __launch_bounds__(256)
k_tcr_post_cols(int n, int rows2, const float2* __restrict__ V, float* __restrict__ PT,
                float* __restrict__ RT) {
    const int groups = rows2 / 4, half = n / 2;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)groups * half) return;
    const int g = (int)(q / half), j = (int)(q % half);
    float4* dp = reinterpret_cast<float4*>(PT + (size_t)j * 2 * n + 16 * g);
    float4* dr4 = reinterpret_cast<float4*>(RT + (size_t)j * 2 * n + 16 * g);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float2* zp = V + (size_t)(4 * g + t) * n;
        const float2* zr = V + (size_t)(rows2 + 4 * g + t) * n;
        const float2 p0 = zp[j], p1 = zp[n - 1 - j], r0 = zr[j], r1 = zr[n - 1 - j];
        dp[t] = make_float4(p0.x, p1.x, p0.y, p1.y);
        dr4[t] = make_float4(r0.x, -r1.x, r0.y, -r1.y);
    }
}

// Inverse inputs of the row pass for y-row pairs r: Z[r] E_x (reversed sine
// coefficients of w_u P), Z[rows2 + r] E_y (cosine sums of R), as the fill
// of k_rows_inv.
__global__ void __launch_bounds__(256)
k_tcr_pack_inv(int n, int rows2, const float* __restrict__ PT, const float* __restrict__ RT,
               const float2* __restrict__ ph, float pi_lx, float2* __restrict__ Z) {
    const int half = n / 2 + 1;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)rows2 * half) return;
    const int r = (int)(q / half), u = (int)(q % half);
    const int un = (n - u) & (n - 1);
    {
        const float2* A = reinterpret_cast<const float2*>(RT) + (size_t)r * n;
        const float2 cu = A[u & (n - 1)], cn = A[un];
        const float au = cu.x, bu = cu.y;
        const float an = (u > 0) ? cn.x : 0.0f, bn = (u > 0) ? cn.y : 0.0f;
        const float cau = (u == 0) ? au : 0.5f * au, cbu = (u == 0) ? bu : 0.5f * bu;
        float can = 0.5f * an, cbn = 0.5f * bn;
        if (u == n / 2) { can = cau; cbn = cbu; }
        float2* row = Z + (size_t)(rows2 + r) * n;
        row[u & (n - 1)] = pack_inv(cau, can, cbu, cbn, ph[u]);
        if (u > 0 && u < n / 2) row[n - u] = pack_inv(can, cau, cbn, cbu, ph[n - u]);
    }
    {
        const float2* Pr = reinterpret_cast<const float2*>(PT) + (size_t)r * n;
        const float2 cu = Pr[u & (n - 1)], cn = Pr[un];
        const float wu = pi_lx * (float)u, wn = pi_lx * (float)(n - u);
        const float ca_u = (u == 0) ? 0.0f : 0.5f * wn * cn.x;
        const float cb_u = (u == 0) ? 0.0f : 0.5f * wn * cn.y;
        float ca_n = (u == 0) ? 0.0f : 0.5f * wu * cu.x;
        float cb_n = (u == 0) ? 0.0f : 0.5f * wu * cu.y;
        if (u == n / 2) { ca_n = ca_u; cb_n = cb_u; }
        float2* row = Z + (size_t)r * n;
        row[u & (n - 1)] = pack_inv(ca_u, ca_n, cb_u, cb_n, ph[u]);
        if (u > 0 && u < n / 2) row[n - u] = pack_inv(ca_n, ca_u, cb_n, cb_u, ph[n - u]);
    }
}

// Inverse outputs of the row pass: E2[y][x] = ((-1)^x E_x, E_y) for the rows
// of pair r, unshuffled.
__global__ void __launch_bounds__(256)
k_tcr_post_rows(int n, int rows2, const float2* __restrict__ V, float2* __restrict__ E2) {
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)rows2 * n) return;
    const int r = (int)(q / n), x = (int)(q % n);
    const int k = mk_src(x, n);
    const float2 zx = V[(size_t)r * n + k], zy = V[(size_t)(rows2 + r) * n + k];
    const float s = (x & 1) ? -1.0f : 1.0f;
    E2[(size_t)(2 * r) * n + x] = make_float2(s * zx.x, zy.x);
    E2[(size_t)(2 * r + 1) * n + x] = make_float2(s * zx.y, zy.y);
}

static inline unsigned tcr_blocks(long long items) { return (unsigned)((items + 255) / 256); }

cudaError_t launch_tcr_stage(Ctx& c, int which, const float2* V, float2* Z, cudaStream_t s) {
    const int n = c.n, rows2 = n / 2;
    const float pi_lx = (float)(M_PI / c.Lx), pi_ly = (float)(M_PI / c.Ly);
    switch (which) {
        case 0: {   // rho rows -> Z (with the overflow and charge sums)
            const float inv_ab = (float)(1.0 / c.Ab);
            const float cap = (float)(c.opt.target_density * c.Ab);
            const unsigned nb = tcr_blocks((long long)rows2 * (n / 2));
            if (c.opt.deterministic)
                k_tcr_pack_rho<true><<<nb, 256, 0, s>>>(n, rows2, nullptr, c.Dq, c.M, inv_ab, cap,
                                                        Z, c.acc, det_red(c, 0));
            else
                k_tcr_pack_rho<false><<<nb, 256, 0, s>>>(n, rows2, c.D, nullptr, c.M, inv_ab, cap,
                                                         Z, c.acc, det_red(c, 0));
            break;
        }
        case 1:     // row spectra -> T1 (transposed)
            k_tcr_post_fwd<<<tcr_blocks((long long)(rows2 / 4) * (n / 2 + 1)), 256, 0, s>>>(
                n, rows2 / 4, V, c.ph, c.T1);
            break;
        case 2:     // T1 rows -> Z
            k_tcr_pack_rows<<<tcr_blocks((long long)rows2 * (n / 2)), 256, 0, s>>>(n, rows2, c.T1, Z);
            break;
        case 3:     // column spectra -> divide, energy -> Z (P rows, then R rows)
            k_tcr_spectral<<<tcr_blocks((long long)rows2 * (n / 2 + 1)), 256, 0, s>>>(
                n, rows2, V, c.ph, pi_lx, pi_ly, (float)c.opt.helmholtz_eps, Z, c.acc,
                det_red(c, 0));
            break;
        case 4:     // P, R sums -> PT, RT (transposed)
            k_tcr_post_cols<<<tcr_blocks((long long)(rows2 / 4) * (n / 2)), 256, 0, s>>>(n, rows2, V,
                                                                                        c.PT, c.RT);
            break;
        case 5:     // PT, RT rows -> Z (E_x rows, then E_y rows)
            k_tcr_pack_inv<<<tcr_blocks((long long)rows2 * (n / 2 + 1)), 256, 0, s>>>(
                n, rows2, c.PT, c.RT, c.ph, pi_lx, Z);
            break;
        default:    // E_x, E_y sums -> E2
            k_tcr_post_rows<<<tcr_blocks((long long)rows2 * n), 256, 0, s>>>(n, rows2, V, c.E2);
            break;
    }
    c.launches++;
    return cudaGetLastError();
}

// ------------------------------------------------------------ launch
enum { PASS_FWD, PASS_COLS, PASS_FIELD, PASS_PSI, PASS_MAPS };

template <int LOGN>
static cudaError_t launch_all_logn(Ctx& c, int which, cudaStream_t s) {
    using L2 = Lay<LOGN, 2>;
    using L1 = Lay<LOGN, 1>;
    constexpr int N = 1 << LOGN;
    constexpr int nb2 = (N / 4 + L2::GB - 1) / L2::GB, nb1 = (N / 2 + L1::GB - 1) / L1::GB;
    const float inv_ab = (float)(1.0 / c.Ab);
    const float cap = (float)(c.opt.target_density * c.Ab);
    const float pi_lx = (float)(M_PI / c.Lx), pi_ly = (float)(M_PI / c.Ly);
    const int tma = c.spec_tma ? 1 : 0;
    auto inv = [&](auto kern, int nv) {
        return launch_chain(kern, nb1, L1::T, L1::GB * L1::group_bytes(nv), s, c.chain, c.PT, c.RT,
                            c.E2, c.psi, c.ex, c.ey, pi_lx);
    };
    cudaError_t e = cudaSuccess;
    switch (which) {
        case PASS_FWD: {
            const int smem = L2::GB * L2::group_bytes(1);
            auto fwd = [&](auto kern) {
                return launch_chain(kern, nb2, L2::T, smem, s, c.chain, c.D, c.Dq, c.M, inv_ab,
                                    cap, c.T1, c.acc, det_red(c, 0), c.map_t1, tma);
            };
            e = c.opt.deterministic ? fwd(k_rows_fwd<LOGN, true>) : fwd(k_rows_fwd<LOGN, false>);
            break;
        }
        case PASS_COLS:
            e = launch_chain(k_cols<LOGN>, nb2, L2::T, L2::GB * L2::group_bytes(2), s, c.chain,
                             c.T1, c.PT, c.RT, pi_lx, pi_ly, (float)c.opt.helmholtz_eps, c.acc,
                             det_red(c, 0), c.map_pt, c.map_rt, tma);
            break;
        case PASS_FIELD: e = inv(k_rows_inv<LOGN, INV_FIELD>, 2); break;
        case PASS_PSI: e = inv(k_rows_inv<LOGN, INV_PSI>, 1); break;
        default: e = inv(k_rows_inv<LOGN, INV_MAPS>, 2); break;
    }
    c.launches++;
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

// Shared-memory opt-in for every kernel of one transform size (done at create,
// outside any stream capture).
template <int LOGN>
static void prepare_logn() {
    using L2 = Lay<LOGN, 2>;
    using L1 = Lay<LOGN, 1>;
    auto set = [](auto kern, int smem) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    };
    set(k_rows_fwd<LOGN, true>, L2::GB * L2::group_bytes(1));
    set(k_rows_fwd<LOGN, false>, L2::GB * L2::group_bytes(1));
    set(k_cols<LOGN>, L2::GB * L2::group_bytes(2));
    set(k_rows_inv<LOGN, INV_FIELD>, L1::GB * L1::group_bytes(2));
    set(k_rows_inv<LOGN, INV_PSI>, L1::GB * L1::group_bytes(1));
    set(k_rows_inv<LOGN, INV_MAPS>, L1::GB * L1::group_bytes(2));
}

void prepare_spectral(int logn) {
    switch (logn) {
        case 4: prepare_logn<4>(); break;
        case 5: prepare_logn<5>(); break;
        case 6: prepare_logn<6>(); break;
        case 7: prepare_logn<7>(); break;
        case 8: prepare_logn<8>(); break;
        case 9: prepare_logn<9>(); break;
        case 10: prepare_logn<10>(); break;
        case 11: prepare_logn<11>(); break;
        case 12: prepare_logn<12>(); break;
        default: break;
    }
}

static cudaError_t dispatch(Ctx& c, int which, cudaStream_t s) {
    switch (c.logn) {
        case 4: return launch_all_logn<4>(c, which, s);
        case 5: return launch_all_logn<5>(c, which, s);
        case 6: return launch_all_logn<6>(c, which, s);
        case 7: return launch_all_logn<7>(c, which, s);
        case 8: return launch_all_logn<8>(c, which, s);
        case 9: return launch_all_logn<9>(c, which, s);
        case 10: return launch_all_logn<10>(c, which, s);
        case 11: return launch_all_logn<11>(c, which, s);
        case 12: return launch_all_logn<12>(c, which, s);
        default: return cudaErrorInvalidValue;
    }
}

void spec_maps_init(Ctx& c) {
    // n/2 rows of n complex elements, boxes of four of them by up to 256 rows
    const int n = c.n, rows = n / 2, box = rows < 256 ? rows : 256;
    c.spec_maps_ok = c.T1 && c.PT && c.RT && n >= 16 &&
                     make_map_f32(&c.map_t1, c.T1, rows, 2 * n, 8, box) &&
                     make_map_f32(&c.map_pt, c.PT, rows, 2 * n, 8, box) &&
                     make_map_f32(&c.map_rt, c.RT, rows, 2 * n, 8, box);
    c.spec_tma = c.spec_maps_ok;
}

cudaError_t launch_rows_fwd(Ctx& c, cudaStream_t s) { return dispatch(c, PASS_FWD, s); }
cudaError_t launch_cols_spectral(Ctx& c, cudaStream_t s) { return dispatch(c, PASS_COLS, s); }
cudaError_t launch_rows_inv(Ctx& c, cudaStream_t s) { return dispatch(c, PASS_FIELD, s); }
cudaError_t launch_rows_psi(Ctx& c, cudaStream_t s) { return dispatch(c, PASS_PSI, s); }
cudaError_t launch_rows_maps(Ctx& c, cudaStream_t s) { return dispatch(c, PASS_MAPS, s); }

}  // namespace fftpl
