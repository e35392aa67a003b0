// Forward passes on the row-group layout: d = A x (dose_spmv), the same with
// FP64 vectors (dose_spmv_f64) and the batched SpMM D_m = A_m X_m for several
// matrices (beams x uncertainty scenarios, Sec. I) and up to 16 spot-weight
// vectors each.
//
// One CTA per SM.  Every worker warp streams its own packets of row groups
// through its own ring of bulk copies (rg_common.cuh), issued before the CTA
// gathers its columns of x into shared memory; one more warp writes the rows
// without entries.  A warp takes one group at a time: lane l handles union
// columns l, l + 32, ... with one column load, one load of the rows' values and
// one gather of x per column, sums all rows of the group in packed FP32 pairs
// and reduces them over the warp with a transposed butterfly.  Static
// assignment and fixed orders: results are bitwise repeatable.
#include "dfloat.cuh"
#include "rg_common.cuh"

#include <algorithm>
#include <type_traits>

namespace dose {
namespace {

constexpr uint32_t kMvWorkers = 24;   // most worker warps of the single-vector form
constexpr uint32_t kMv64Workers = 16; // ... of the FP64-vector form
// worker warps of the batched form: the second where the first leaves no room
// for the window of X (all matrices of a launch share them)
constexpr uint32_t kMmWorkers[2] = {12, 6};

// Shared memory before the rings: header, zeros, the CTA's columns of x.
size_t fwd_fixed(uint32_t wmax, uint32_t x_bytes) {
    return kRgHeader + kRgZeroBytes + ((size_t)(wmax + 1) * x_bytes + 127) / 128 * 128;
}
// X of the batched form: blocks of 8 columns (see mm_x).
size_t mm_fixed(uint32_t wmax, uint32_t nq) { return kRgHeader + kRgZeroBytes + (size_t)(wmax + 8) / 8 * 128 * nq; }

struct FwdParams {
    RgView A;
    const void* x;
    void* d;
    uint32_t wmax, nw, depth, slot;
    int* err;
};

// Bound by memory and issue alike: 1.5e8 entries (u16, 16-bit columns, 408 MB of its
// own bytes) take 66.3 us, 0.90 of 6.8 TB/s, against 109.6 us with groups of four
// consecutive rows (488 MB, 0.66) and one ring of stages for all warps of a CTA: eight
// rows share each column and each x, so a third of the instructions went, and a warp
// never waits for the others' packets.
template <int FMT, int HR, uint32_t IW>
__global__ void __launch_bounds__((kMvWorkers + 1) * 32, 1) rg_spmv_kernel(const __grid_constant__ FwdParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NW = p.nw;
    unsigned char* zeros = smem + kRgHeader;
    float* xs = reinterpret_cast<float*>(zeros + kRgZeroBytes);
    unsigned char* slot_base = reinterpret_cast<unsigned char*>(xs) + round_up((p.wmax + 1) * 4, 128);
    const uint32_t cta = blockIdx.x, T = blockDim.x, t = threadIdx.x;
    rg_let_next_start();
    RgStream<RG_FORWARD> S;
    RgDict C;
    C.range(p.A, cta);
    if (warp < NW) S.range(p.A, cta, NW, warp);
    C.load(t, T);
    if (warp < NW) {
        S.entry();
        S.start(warp, p.depth, p.slot, smem, slot_base, lane);
    }
    const uint32_t nc = C.nc;
    rg_wait_previous();
    C.each(t, T, [&](uint32_t c) { return __ldcg(static_cast<const float*>(p.x) + c); },
           [&](uint32_t j, float v) { xs[j] = v; });
    if (t == 0) xs[nc] = 0.f;
    __syncthreads();
    float* __restrict__ d = static_cast<float*>(p.d);
    if (warp >= NW) {
        rg_fill_zeros(zeros, lane);
        rg_zero_rows(p.A.zero_runs, p.A.n_zero_runs, static_cast<unsigned char*>(p.d), 4, zeros, lane);
        return;
    }
    uint64_t acc[HR / 2];
    while (S.pending) {
        if (!S.wait(p.err)) return;
        const RgSlotView<FMT, HR, IW> P(S.slot());
        if (rg_packet_ok(P, S.slot(), p.slot, p.A.nrows, nc, lane, p.err)) {
            const uint32_t fl = S.flag();
            uint32_t u = 0;
            for (uint32_t g = 0; g < P.ng; ++g) {
                const uint32_t n = P.gn[g];
                const uint32_t row = P.rows[g * HR + lane / (32 / HR)];
                if (!(fl & RG_CARRY_IN)) {
#pragma unroll
                    for (int i = 0; i < HR / 2; ++i) acc[i] = 0ull;
                }
                rg_dot<FMT, HR, IW>(P.cols + u * IW, P.vals + u * RgVal<FMT, HR>::kBytes, n, lane, xs, nc, acc);
                u += n;
                if (fl & RG_CARRY_OUT) continue;
                const float sum = rg_reduce<HR>(acc, lane);
                if ((lane & (32 / HR - 1)) == 0 && row != 0xFFFFFFFFu) {
                    float sc = p.A.scale;
                    if (FMT == DOSE_FMT_FP8E4M3_ROWSCALE) sc = P.scales[g * HR + lane / (32 / HR)];
                    d[row] = FMT == DOSE_FMT_FP8E4M3_ROWSCALE || FMT == DOSE_FMT_U16_SCALE ? __fmul_rn(sc, sum) : sum;
                }
            }
        }
        S.done(lane);
    }
}

// ---- FP64 vectors (dose_spmv_f64)

// HR rows' accumulators of one lane: double-float pairs as packed FP32 (rows
// 2 i, 2 i + 1 in one register pair: the operations of df_mac, two rows at a
// time), or doubles.
template <int MODE, int HR>
struct Acc64;
template <int HR>
struct Acc64<F64_DF, HR> {
    uint64_t s[HR / 2], c[HR / 2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < HR / 2; ++i) s[i] = c[i] = 0ull;
    }
    template <class V>
    __device__ __forceinline__ void mac(const V& q, uint2 x) {
        const uint64_t hi = dev::f2_pack(x.x, x.x), lo = dev::f2_pack(x.y, x.y), m1 = dev::f2_splat(-1.0f);
        const uint64_t nhi = dev::f2_mul(hi, m1);
#pragma unroll
        for (int i = 0; i < HR / 2; ++i) {
            const uint64_t a = q.pair(i);
            const uint64_t np = dev::f2_mul(a, nhi);  // -p, p = fl(a hi)
            const uint64_t e = dev::f2_fma(a, lo, dev::f2_fma(a, hi, np));
            // TwoSum(s, p); a difference u - v is fma(v, -1, u), rounded as u - v is
            const uint64_t t = dev::f2_fma(np, m1, s[i]);
            const uint64_t bp = dev::f2_fma(s[i], m1, t);
            const uint64_t as = dev::f2_fma(dev::f2_fma(bp, m1, t), m1, s[i]);
            const uint64_t err = dev::f2_fma(dev::f2_add(np, bp), m1, as);
            s[i] = t;
            c[i] = dev::f2_add(c[i], dev::f2_add(err, e));
        }
    }
    // row l / (32 / HR)'s total in lane l
    __device__ __forceinline__ Acc<F64_DF> reduce(uint32_t lane) const {
        Acc<F64_DF> a[HR];
#pragma unroll
        for (int i = 0; i < HR / 2; ++i) {
            dev::f2_split(s[i], a[2 * i].s, a[2 * i + 1].s);
            dev::f2_split(c[i], a[2 * i].c, a[2 * i + 1].c);
        }
        return fold(a, lane);
    }
    __device__ __forceinline__ static Acc<F64_DF> fold(Acc<F64_DF> (&a)[HR], uint32_t lane) {
        uint32_t o = 16;
#pragma unroll
        for (int n = HR / 2; n >= 1; n /= 2, o /= 2) {
            const bool hi = lane & o;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                Acc<F64_DF> keep, send;
                keep.s = hi ? a[i + n].s : a[i].s;
                keep.c = hi ? a[i + n].c : a[i].c;
                send.s = hi ? a[i].s : a[i + n].s;
                send.c = hi ? a[i].c : a[i + n].c;
                keep.add(send.shfl_xor(o));
                a[i] = keep;
            }
        }
        for (; o > 0; o /= 2) a[0].add(a[0].shfl_xor(o));
        return a[0];
    }
};
template <int HR>
struct Acc64<F64_DP, HR> {
    double v[HR];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < HR; ++i) v[i] = 0.0;
    }
    template <class V>
    __device__ __forceinline__ void mac(const V& q, uint2 x) {
        const double xd = __hiloint2double((int)x.y, (int)x.x);
#pragma unroll
        for (int i = 0; i < HR / 2; ++i) {
            float a0, a1;
            dev::f2_split(q.pair(i), a0, a1);
            v[2 * i] = __fma_rn((double)a0, xd, v[2 * i]);
            v[2 * i + 1] = __fma_rn((double)a1, xd, v[2 * i + 1]);
        }
    }
    __device__ __forceinline__ Acc<F64_DP> reduce(uint32_t lane) const {
        double a[HR];
#pragma unroll
        for (int i = 0; i < HR; ++i) a[i] = v[i];
        uint32_t o = 16;
#pragma unroll
        for (int n = HR / 2; n >= 1; n /= 2, o /= 2) {
            const bool hi = lane & o;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const double keep = hi ? a[i + n] : a[i], send = hi ? a[i] : a[i + n];
                a[i] = __dadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, o));
            }
        }
        for (; o > 0; o /= 2) a[0] = __dadd_rn(a[0], __shfl_xor_sync(0xffffffffu, a[0], o));
        Acc<F64_DP> r;
        r.v = a[0];
        return r;
    }
};

// Bound by the FP32 pair arithmetic (issue 63 % active, memory 42 %), so one packed
// instruction does two rows' step: 6.3e7 F16 entries take 60.0 us, against 111.5 us
// entry by entry on CSR (twice the instructions and 2.5 times the bytes).  16 warps:
// the pairs of eight rows take 94 registers a thread.
template <int FMT, int HR, uint32_t IW, int MODE>
__global__ void __launch_bounds__((kMv64Workers + 1) * 32, 1) rg_spmv64_kernel(const __grid_constant__ FwdParams p) {
    constexpr uint32_t VB = RgVal<FMT, HR>::kBytes;
    extern __shared__ __align__(128) unsigned char smem[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NW = p.nw;
    unsigned char* zeros = smem + kRgHeader;
    uint2* xs = reinterpret_cast<uint2*>(zeros + kRgZeroBytes);
    unsigned char* slot_base = reinterpret_cast<unsigned char*>(xs) + round_up((p.wmax + 1) * 8, 128);
    const uint32_t cta = blockIdx.x, T = blockDim.x, t = threadIdx.x;
    rg_let_next_start();
    RgStream<RG_FORWARD> S;
    RgDict C;
    C.range(p.A, cta);
    if (warp < NW) S.range(p.A, cta, NW, warp);
    C.load(t, T);
    if (warp < NW) {
        S.entry();
        S.start(warp, p.depth, p.slot, smem, slot_base, lane);
    }
    const uint32_t nc = C.nc;
    rg_wait_previous();
    C.each(t, T, [&](uint32_t c) { return __ldcg(static_cast<const double*>(p.x) + c); },
           [&](uint32_t j, double v) { xs[j] = prepare_x<MODE>(v); });
    if (t == 0) xs[nc] = make_uint2(0u, 0u);
    __syncthreads();
    if (warp >= NW) {
        rg_fill_zeros(zeros, lane);
        rg_zero_rows(p.A.zero_runs, p.A.n_zero_runs, static_cast<unsigned char*>(p.d), 8, zeros, lane);
        return;
    }
    double* __restrict__ d = static_cast<double*>(p.d);
    Acc64<MODE, HR> acc;
    while (S.pending) {
        if (!S.wait(p.err)) return;
        const RgSlotView<FMT, HR, IW> P(S.slot());
        if (rg_packet_ok(P, S.slot(), p.slot, p.A.nrows, nc, lane, p.err)) {
            const uint32_t fl = S.flag();
            uint32_t u0 = 0;
            for (uint32_t g = 0; g < P.ng; ++g) {
                const uint32_t n = P.gn[g];
                const uint32_t row = P.rows[g * HR + lane / (32 / HR)];
                const unsigned char* cols = P.cols + u0 * IW;
                const unsigned char* vals = P.vals + u0 * VB;
                u0 += n;
                if (!(fl & RG_CARRY_IN)) acc.zero();
#pragma unroll 2
                for (uint32_t u = lane; u < round_up(n, 32); u += 32) {
                    RgVal<FMT, HR> q;
                    uint32_t c = nc;
                    q.zero();
                    if (u < n) {
                        c = rg_col<IW>(cols, u);
                        q.load(vals + u * VB);
                    }
                    acc.mac(q, xs[c]);
                }
                if (fl & RG_CARRY_OUT) continue;
                const Acc<MODE> tot = acc.reduce(lane);
                if ((lane & (32 / HR - 1)) == 0 && row != 0xFFFFFFFFu) {
                    float sc = p.A.scale;
                    if (FMT == DOSE_FMT_FP8E4M3_ROWSCALE) sc = P.scales[g * HR + lane / (32 / HR)];
                    d[row] = tot.result(FMT == DOSE_FMT_FP8E4M3_ROWSCALE || FMT == DOSE_FMT_U16_SCALE, sc);
                }
            }
        }
        S.done(lane);
    }
}

// ---- batched SpMM

struct MmItem {
    RgView A;
    const float* X;  // ncols x nvec, row-major
    float* D;        // nrows x nvec, row-major
};

struct MmParams {
    MmItem item[kRgSpmmMaxPerLaunch];
    uint32_t count, nvec, nw, depth, slot, wmax;
    int* err;
};

// Word offset of 4 q (vector quad q) of local column c in the staged window of
// X: blocks of 8 columns, in each NQ rows of 128 bytes holding quad q of the 8
// columns, so that 8 lanes reading one quad of 8 columns that differ mod 8
// touch 8 distinct bank quads.
template <int NQ>
__device__ __forceinline__ uint32_t mm_x(uint32_t c, uint32_t q) {
    return (c >> 3) * (32 * NQ) + q * 32 + (c & 7u) * 4;
}

// Lane l: vector quad q = l / S, union columns u = s, s + S, ... (s = l mod S,
// S = 32 / NQ); per column the HR rows' values in one load, one 16-byte X load
// and 2 HR packed FMAs (rows 2 i and 2 i + 1 times one vector's weight).  NQ =
// quads of vectors (1, 2 or 4): fewer vectors put more lanes on the columns
// instead of computing vectors nobody asked for.
// Bound by issue (47 % active) and the spread of the CTAs' times (mean 84 % of the
// longest): 16 vectors times three matrices (160 x 160 x 80 voxels, 1000 spots) take
// 138.4 us, 172.9 with groups of four rows, whose X loads were twice as many and kept
// the shared memory 56 % busy (33 % now); 5 vectors times two matrices 36.6 us, 96.9
// when 16 were always computed.  12 warps: 96 registers a thread.
template <int FMT, int HR, uint32_t IW, int NQ>
__global__ void __launch_bounds__((kMmWorkers[0] + 1) * 32, 1) rg_spmm_kernel(const __grid_constant__ MmParams p) {
    constexpr uint32_t VB = RgVal<FMT, HR>::kBytes;
    constexpr uint32_t SL = 32 / NQ;
    extern __shared__ __align__(128) unsigned char smem[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* zeros = smem + kRgHeader;
    float* xs = reinterpret_cast<float*>(zeros + kRgZeroBytes);
    unsigned char* slot_base = reinterpret_cast<unsigned char*>(xs) + (p.wmax + 8) / 8 * 128 * NQ;
    rg_let_next_start();
    if (warp >= p.nw) {
        rg_fill_zeros(zeros, lane);
        rg_wait_previous();
        for (uint32_t m = 0; m < p.count; ++m)
            rg_zero_rows(p.item[m].A.zero_runs, p.item[m].A.n_zero_runs, reinterpret_cast<unsigned char*>(p.item[m].D),
                         4 * p.nvec, zeros, lane);
        return;
    }
    const uint32_t nct = p.nw * 32, q = lane / SL, s = lane % SL;
    RgStream<RG_FORWARD> S;
    bool ok = true;  // after a timeout the warp stays for the barriers but takes no more packets
    for (uint32_t m = 0; m < p.count; ++m) {
        const MmItem& it = p.item[m];
        // A CTA's shares of different matrices come from different places of the
        // row order (0.382 of the grid apart): a share is cut for the single-vector
        // kernels, whose cost per group is higher, so shares of the beam's centre
        // (long unions) take longer here than shares of its edge.
        const uint32_t cta = (blockIdx.x + m * (uint32_t)(0.382f * gridDim.x)) % gridDim.x;
        RgDict C;
        C.range(it.A, cta);
        if (ok) {
            S.range(it.A, cta, p.nw, warp);
            S.entry();
            if (m)
                S.fill(lane);
            else
                S.start(warp, p.depth, p.slot, smem, slot_base, lane);
        }
        const uint32_t nc = C.nc;
        if (m)
            dev::named_barrier(1, nct);  // every worker is done with the previous window of X
        else
            rg_wait_previous();
        for (uint32_t j = threadIdx.x; j < (nc + 1) * 4 * NQ; j += nct) {
            const uint32_t c = j / (4 * NQ), v = j % (4 * NQ);
            xs[mm_x<NQ>(c, v >> 2) + (v & 3u)] =
                c < nc && v < p.nvec ? __ldcg(it.X + (size_t)__ldg(C.dict + c) * p.nvec + v) : 0.f;
        }
        dev::named_barrier(1, nct);
        const bool vec4 = (p.nvec & 3u) == 0 && (reinterpret_cast<uintptr_t>(it.D) & 15u) == 0;
        uint64_t acc[HR / 2][4];  // rows 2 i, 2 i + 1 and vectors 4 q + v
        while (S.pending) {
            if (!(ok = S.wait(p.err))) break;
            const RgSlotView<FMT, HR, IW> P(S.slot());
            if (rg_packet_ok(P, S.slot(), p.slot, it.A.nrows, nc, lane, p.err)) {
                const uint32_t fl = S.flag();
                uint32_t u0 = 0;
                for (uint32_t g = 0; g < P.ng; ++g) {
                    const uint32_t n = P.gn[g];
                    const unsigned char* cols = P.cols + u0 * IW;
                    const unsigned char* vals = P.vals + u0 * VB;
                    u0 += n;
                    if (!(fl & RG_CARRY_IN)) {
#pragma unroll
                        for (int i = 0; i < HR / 2; ++i)
#pragma unroll
                            for (int v = 0; v < 4; ++v) acc[i][v] = 0ull;
                    }
                    auto mac = [&](const RgVal<FMT, HR>& w, uint32_t c) {
                        const float4 x = *reinterpret_cast<const float4*>(xs + mm_x<NQ>(c, q));
                        const uint64_t x0 = dev::f2_splat(x.x), x1 = dev::f2_splat(x.y), x2 = dev::f2_splat(x.z),
                                       x3 = dev::f2_splat(x.w);
#pragma unroll
                        for (int i = 0; i < HR / 2; ++i) {
                            const uint64_t a = w.pair(i);
                            acc[i][0] = dev::f2_fma(a, x0, acc[i][0]);
                            acc[i][1] = dev::f2_fma(a, x1, acc[i][1]);
                            acc[i][2] = dev::f2_fma(a, x2, acc[i][2]);
                            acc[i][3] = dev::f2_fma(a, x3, acc[i][3]);
                        }
                    };
                    const uint32_t nfull = n / SL;
                    uint32_t u = s;
#pragma unroll 2
                    for (uint32_t k = 0; k < nfull; ++k, u += SL) {
                        RgVal<FMT, HR> w;
                        w.load(vals + u * VB);
                        mac(w, rg_col<IW>(cols, u));
                    }
                    if (n % SL) {
                        RgVal<FMT, HR> w;
                        uint32_t c = nc;
                        w.zero();
                        if (u < n) {
                            c = rg_col<IW>(cols, u);
                            w.load(vals + u * VB);
                        }
                        mac(w, c);
                    }
                    if (fl & RG_CARRY_OUT) continue;
                    // sum over the slices s: a transposed butterfly over the rows, then
                    // (more slices than rows) plain additions; lane s ends with row
                    // s / (SL / HR), vectors 4 q .. 4 q + 3
                    float a[HR][4];
#pragma unroll
                    for (int i = 0; i < HR / 2; ++i)
#pragma unroll
                        for (int v = 0; v < 4; ++v) dev::f2_split(acc[i][v], a[2 * i][v], a[2 * i + 1][v]);
                    uint32_t o = SL / 2;
#pragma unroll
                    for (int h = HR / 2; h >= 1; h /= 2, o /= 2) {
                        const bool hi = lane & o;
#pragma unroll
                        for (int i = 0; i < h; ++i)
#pragma unroll
                            for (int v = 0; v < 4; ++v) {
                                const float keep = hi ? a[i + h][v] : a[i][v], send = hi ? a[i][v] : a[i + h][v];
                                a[i][v] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, o));
                            }
                    }
                    for (; o > 0; o /= 2)
#pragma unroll
                        for (int v = 0; v < 4; ++v)
                            a[0][v] = __fadd_rn(a[0][v], __shfl_xor_sync(0xffffffffu, a[0][v], o));
                    const uint32_t gr = g * HR + s / (SL / HR), row = P.rows[gr];
                    if (s % (SL / HR) == 0 && row != 0xFFFFFFFFu) {
                        float sc = it.A.scale;
                        if (FMT == DOSE_FMT_FP8E4M3_ROWSCALE) sc = P.scales[gr];
                        if (FMT == DOSE_FMT_FP8E4M3_ROWSCALE || FMT == DOSE_FMT_U16_SCALE) {
#pragma unroll
                            for (int v = 0; v < 4; ++v) a[0][v] = __fmul_rn(sc, a[0][v]);
                        }
                        float* dr = it.D + (size_t)row * p.nvec + 4 * q;
                        if (vec4) {
                            if (4 * q < p.nvec) *reinterpret_cast<float4*>(dr) = make_float4(a[0][0], a[0][1], a[0][2], a[0][3]);
                        } else {
#pragma unroll
                            for (uint32_t v = 0; v < 4; ++v)
                                if (4 * q + v < p.nvec) dr[v] = a[0][v];
                        }
                    }
                }
            }
            S.done(lane);
        }
    }
}

// ---- launches

// Calls f(format, rows per group, index width) as compile-time constants.
template <int V>
using Int = std::integral_constant<int, V>;
template <int FMT, class F>
cudaError_t by_shape(const RowGroups& R, F f) {
    if (value_bytes(FMT) <= 2 && R.hr == 8) {
        constexpr int H = value_bytes(FMT) <= 2 ? 8 : 4;
        return R.iw == 2 ? f(Int<FMT>{}, Int<H>{}, Int<2>{}) : f(Int<FMT>{}, Int<H>{}, Int<4>{});
    }
    return R.iw == 2 ? f(Int<FMT>{}, Int<4>{}, Int<2>{}) : f(Int<FMT>{}, Int<4>{}, Int<4>{});
}
template <class F>
cudaError_t by_format(const dose_matrix* A, F f) {
    switch (A->fmt) {
        case DOSE_FMT_U16_SCALE: return by_shape<DOSE_FMT_U16_SCALE>(A->rg, f);
        case DOSE_FMT_BF16: return by_shape<DOSE_FMT_BF16>(A->rg, f);
        case DOSE_FMT_F16: return by_shape<DOSE_FMT_F16>(A->rg, f);
        case DOSE_FMT_F32: return by_shape<DOSE_FMT_F32>(A->rg, f);
        case DOSE_FMT_FP8E4M3_ROWSCALE: return by_shape<DOSE_FMT_FP8E4M3_ROWSCALE>(A->rg, f);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// Worker warps of a forward pass that fit: as many as the form takes while two
// slots each fit beside the CTA's columns of x, then as deep rings as fit.
uint32_t rg_forward_warps(const dose_matrix* A, int which, uint32_t* depth, size_t* smem) {
    const RowGroups& R = A->rg;
    if (!R.built) return 0;
    // (whether the batched form fits depends on the other matrices of a call: rg_spmm_applies)
    if (which == RG_DEAL_SPMM || which == RG_DEAL_SPMM_FEW) return kMmWorkers[which == RG_DEAL_SPMM_FEW];
    const uint32_t xb = which == RG_DEAL_F64 ? 8 : 4, most = which == RG_DEAL_F64 ? kMv64Workers : kMvWorkers;
    const size_t fixed = fwd_fixed(R.wmax, xb);
    if (fixed + 2ull * R.slot > kMaxSmemPerBlock) return 0;
    const uint32_t nw = (uint32_t)std::min<size_t>(most, (kMaxSmemPerBlock - fixed) / (2ull * R.slot));
    const uint32_t d = (uint32_t)std::min<size_t>(kRgMaxDepth, (kMaxSmemPerBlock - fixed) / ((size_t)nw * R.slot));
    if (depth) *depth = d;
    if (smem) *smem = fixed + (size_t)nw * d * R.slot;
    return nw;
}

// One launch of the batched form: the matrices A[k] (k in [first, count)) whose
// groups hold hr rows, at most kRgSpmmMaxPerLaunch of them.  Returns how many
// (idx: which), *next the first k not looked at.
static int mm_take(const dose_matrix* const* A, int count, int first, uint32_t hr, int* idx, int* next) {
    int n = 0, k = first;
    for (; k < count && n < (int)kRgSpmmMaxPerLaunch; ++k)
        if (A[k]->rg.hr == hr && A[k]->nrows) idx[n++] = k;
    *next = k;
    return n;
}

// Warps, ring depth and shared memory of a launch over the matrices idx[0 .. n):
// false if the widest window of X (nq quads of vectors) and two slots per warp
// do not fit.
static bool mm_shape(const dose_matrix* const* A, const int* idx, int n, uint32_t nq, MmParams* p, size_t* smem) {
    p->wmax = p->slot = 0;
    for (int i = 0; i < n; ++i) {
        p->wmax = std::max(p->wmax, A[idx[i]]->rg.wmax);
        p->slot = std::max(p->slot, A[idx[i]]->rg.slot);
    }
    const size_t fixed = mm_fixed(p->wmax, nq);
    for (uint32_t nw : kMmWorkers) {
        if (fixed + 2ull * nw * p->slot > kMaxSmemPerBlock) continue;
        p->nw = nw;
        p->depth = (uint32_t)std::min<size_t>(kRgMaxDepth, (kMaxSmemPerBlock - fixed) / ((size_t)nw * p->slot));
        *smem = fixed + (size_t)nw * p->depth * p->slot;
        return true;
    }
    return false;
}

// The row-group form of dose_spmv_batched applies when every matrix has its
// row-group layout (not switched off with adj_layout = 1), all share one stored
// format, index width and grid, and every launch's widest window of X fits
// (whatever the number of vectors).  *launches: kernels of one call.
bool rg_spmm_applies(const dose_matrix* const* A, int count, int* launches) {
    if (count < 1) return false;
    for (int m = 0; m < count; ++m) {
        const RowGroups& R = A[m]->rg;
        if (!R.built || A[m]->adj_tuning.layout == 1) return false;
        if (A[m]->fmt != A[0]->fmt || R.iw != A[0]->rg.iw || R.grid != A[0]->rg.grid) return false;
    }
    int total = 0;
    MmParams p;
    for (uint32_t hr : {8u, 4u})
        for (int k = 0; k < count;) {
            int idx[kRgSpmmMaxPerLaunch];
            size_t smem = 0;
            const int n = mm_take(A, count, k, hr, idx, &k);
            if (!n) continue;
            if (!mm_shape(A, idx, n, 4, &p, &smem)) return false;
            ++total;
        }
    if (launches) *launches = total;
    return true;
}

cudaError_t launch_rg_spmm(const dose_matrix* const* A, int count, const float* const* X, float* const* D, int nvec,
                           cudaStream_t s) {
    const uint32_t nq = nvec <= 4 ? 1 : nvec <= 8 ? 2 : 4;
    for (uint32_t hr : {8u, 4u})
        for (int k = 0; k < count;) {
            int idx[kRgSpmmMaxPerLaunch];
            size_t smem = 0;
            MmParams p;
            const int n = mm_take(A, count, k, hr, idx, &k);
            if (!n) continue;
            if (!mm_shape(A, idx, n, nq, &p, &smem)) return cudaErrorInvalidConfiguration;
            p.count = (uint32_t)n;
            p.nvec = (uint32_t)nvec;
            p.err = A[idx[0]]->err;
            const int which = p.nw == kMmWorkers[0] ? RG_DEAL_SPMM : RG_DEAL_SPMM_FEW;
            for (int i = 0; i < n; ++i) p.item[i] = {rg_view(A[idx[i]], which), X[idx[i]], D[idx[i]]};
            const dose_matrix* M = A[idx[0]];
            const cudaError_t e = by_format(M, [&](auto F, auto H, auto I) {
                constexpr int f = decltype(F)::value, h = decltype(H)::value, iw = decltype(I)::value;
                const uint32_t th = 32 * (p.nw + 1);
                if (nq == 1) return rg_launch(rg_spmm_kernel<f, h, iw, 1>, p, M->rg.grid, th, smem, s);
                if (nq == 2) return rg_launch(rg_spmm_kernel<f, h, iw, 2>, p, M->rg.grid, th, smem, s);
                return rg_launch(rg_spmm_kernel<f, h, iw, 4>, p, M->rg.grid, th, smem, s);
            });
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

static bool fwd_params(const dose_matrix* A, int which, const void* x, void* d, FwdParams* p, size_t* smem) {
    p->nw = rg_forward_warps(A, which, &p->depth, smem);
    if (!p->nw || A->rg.deal[which].nw != p->nw) return false;
    p->A = rg_view(A, which);
    p->x = x;
    p->d = d;
    p->wmax = A->rg.wmax;
    p->slot = A->rg.slot;
    p->err = A->err;
    return true;
}

cudaError_t launch_rg_spmv(const dose_matrix* A, const float* x, float* d, cudaStream_t s) {
    FwdParams p;
    size_t smem = 0;
    if (!fwd_params(A, RG_DEAL_SPMV, x, d, &p, &smem)) return cudaErrorInvalidConfiguration;
    if (A->nrows == 0) return cudaSuccess;
    return by_format(A, [&](auto F, auto H, auto I) {
        return rg_launch(rg_spmv_kernel<decltype(F)::value, decltype(H)::value, decltype(I)::value>, p, A->rg.grid,
                      32 * (p.nw + 1), smem, s);
    });
}

// dose_spmv by default needs three warps beside the CTA's columns of x (51,000 of them):
// 60,000 rows of 300 scattered entries take 95 us with five warps (46,800 columns) and
// 203 us on CSR, so about 160 us with three and 240 with two.
bool rg_spmv_applies(const dose_matrix* A) {
    return rg_forward_warps(A, RG_DEAL_SPMV, nullptr, nullptr) >= (A->fwd.tuning.layout == 2 ? 1u : 3u);
}

// dose_spmv_f64 by default: the arithmetic bounds it, and row groups pay it for every
// stored value, CSR for every entry (2.4 times as much, and a launch).  200 x 200 x 120
// beam with some entries taken out, F16, stored values per entry 1.08 / 2.05 / 2.64 /
// 3.06: 61 / 80 / 81 / 71 us against 112 / 89 / 75 / 49 on CSR; FP8 and F32 alike.  On
// small matrices the launch decides (2e6 entries' worth).  Fewer than 14 warps beside
// the columns of x (8 bytes each) cost about (warps + 2) / 16: 120,000 rows of 300
// scattered entries, eight alike, with 14 / 9 / 6 / 4 / 3 warps 36 / 52 / 68 / 88 / 111
// us, 83 to 95 on CSR.
bool rg_spmv64_applies(const dose_matrix* A) {
    const uint64_t nw = rg_forward_warps(A, RG_DEAL_F64, nullptr, nullptr);
    if (!nw || A->fwd.tuning.layout == 2) return nw > 0;
    const uint64_t stored = A->rg.n_union * A->rg.hr;
    return 16 * stored <= (std::min<uint64_t>(nw, 14) + 2) * (A->nnz * 12ull / 5 + 2000000);
}

cudaError_t launch_rg_spmv64(const dose_matrix* A, const double* x, double* d, bool native, cudaStream_t s) {
    FwdParams p;
    size_t smem = 0;
    if (!fwd_params(A, RG_DEAL_F64, x, d, &p, &smem)) return cudaErrorInvalidConfiguration;
    if (A->nrows == 0) return cudaSuccess;
    return by_format(A, [&](auto F, auto H, auto I) {
        constexpr int f = decltype(F)::value, h = decltype(H)::value, iw = decltype(I)::value;
        const uint32_t th = 32 * (p.nw + 1);
        return native ? rg_launch(rg_spmv64_kernel<f, h, iw, F64_DP>, p, A->rg.grid, th, smem, s)
                      : rg_launch(rg_spmv64_kernel<f, h, iw, F64_DF>, p, A->rg.grid, th, smem, s);
    });
}

}  // namespace dose
