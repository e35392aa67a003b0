// Pieces shared by the row-group kernels (rg_spmm.cu: dose_spmv, dose_spmv_f64
// and the batched SpMM; rg_kernel.cu: adjoint and fused pass): a warp's own
// stream of packets, the packet's parts, the decoders of stored values into
// packed FP32 pairs, and the row sums' butterfly.  The layout is described at
// RowGroups in dose_internal.cuh and rg_layout.cu.
#pragma once

#include "stage_common.cuh"

namespace dose {

// Kernel-side view of one matrix.
struct RgView {
    const unsigned char* data;
    const uint4* pk;
    const uint32_t* row_list;
    const uint32_t* deal;  // of this call
    const uint32_t* dict;
    const uint32_t* dict_begin;
    const uint2* zero_runs;
    uint32_t n_zero_runs, nrows;
    float scale;
};

constexpr uint32_t kRgHeader = 2048;       // 32 warps x 4 mbarriers, then as many packet flag words
constexpr uint32_t kRgMaxDepth = 4;        // ring slots of a warp
constexpr uint32_t kRgZeroBytes = 4096;    // zeros that the bulk stores of rows without entries read

// A row-group kernel's launch, as a programmatic dependent of what is before it
// in the stream (early) or an ordinary one.
template <class K, class P>
cudaError_t rg_launch(K k, const P& p, dim3 grid, uint32_t threads, size_t smem, cudaStream_t s, bool early = true) {
    if (smem > 48 * 1024) {
        const cudaError_t e = allow_max_smem(k);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, p);
}

inline RgView rg_view(const dose_matrix* A, int which) {
    const RowGroups& R = rg_of(A, which);
    RgView v;
    v.data = R.data;
    v.pk = R.deal[which].pk;
    v.row_list = R.row_list;
    v.deal = R.deal[which].begin;
    v.dict = R.dict;
    v.dict_begin = R.dict_begin;
    v.zero_runs = R.zero_runs;
    v.n_zero_runs = R.n_zero_runs;
    v.nrows = A->nrows;
    v.scale = A->fmt == DOSE_FMT_U16_SCALE ? A->scale : 1.0f;
    return v;
}

#ifdef __CUDACC__

namespace dev {
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
                 : "memory");
}
// All bulk stores of this thread done (source read and data written).
__device__ __forceinline__ void bulk_store_wait() {
    asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group 0;" ::: "memory");
}
}  // namespace dev

// ---- programmatic dependent launch.  Every row-group kernel lets the next one
// in its stream start as SMs fall free, and does what depends on the matrix
// alone (ring set-up, the first packets' copies, the column list) before it
// waits for the kernels before it: x and the other vectors are read, and
// results written, only after rg_wait_previous().  Back-to-back calls then hide
// the launch and the first loads' latency (3 to 5 us a call).
// The caller's vectors may thus be written while a kernel that reads them is
// already running: they are read by ordinary loads after the wait (which the
// compiler does not move across it), never through the read-only path, whose data
// must not change while the kernel runs.  x, which a projected-gradient step
// rewrites in place, is read past L1.
__device__ __forceinline__ void rg_let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void rg_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The CTA's columns: the first two of each thread, loaded ahead of the wait.
struct RgDict {
    const uint32_t* dict;
    uint32_t db, nc, c[2];
    __device__ __forceinline__ void range(const RgView& v, uint32_t cta) {
        db = __ldg(v.dict_begin + cta);
        nc = __ldg(v.dict_begin + cta + 1) - db;
        dict = v.dict + db;
    }
    __device__ __forceinline__ void load(uint32_t t, uint32_t nt) {
#pragma unroll
        for (uint32_t k = 0; k < 2; ++k) c[k] = t + k * nt < nc ? __ldg(dict + t + k * nt) : 0u;
    }
    // put(j, get(column)) for this thread's columns j = t, t + nt, ...; four columns,
    // then four values in flight past the first two (a list of 25,000 columns is
    // some thirty rounds of both)
    template <class G, class P>
    __device__ __forceinline__ void each(uint32_t t, uint32_t nt, G get, P put) const {
        decltype(get(0u)) v[4];
#pragma unroll
        for (uint32_t k = 0; k < 2; ++k)
            if (t + k * nt < nc) put(t + k * nt, get(c[k]));
        for (uint32_t j = t + 2 * nt; j < nc; j += 4 * nt) {
            uint32_t q[4];
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) q[k] = __ldg(dict + min(j + k * nt, nc - 1));
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) v[k] = get(q[k]);
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k)
                if (j + k * nt < nc) put(j + k * nt, v[k]);
        }
    }
};

// ---- stored values: HR rows' values of one union column, HR * element size
// bytes (4, 8 or 16), as raw words and as HR / 2 packed FP32 pairs (exact).
template <int FMT, int HR>
struct RgVal {
    static constexpr uint32_t kBytes = HR * (uint32_t)sizeof(typename Fmt<FMT>::T);
    static constexpr uint32_t kWords = kBytes / 4;
    uint32_t w[kWords];

    __device__ __forceinline__ void load(const unsigned char* p) {
        if constexpr (kWords == 4) {
            const uint4 q = *reinterpret_cast<const uint4*>(p);
            w[0] = q.x;
            w[1] = q.y;
            w[2] = q.z;
            w[3] = q.w;
        } else if constexpr (kWords == 2) {
            const uint2 q = *reinterpret_cast<const uint2*>(p);
            w[0] = q.x;
            w[1] = q.y;
        } else {
            w[0] = *reinterpret_cast<const uint32_t*>(p);
        }
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (uint32_t i = 0; i < kWords; ++i) w[i] = 0u;
    }
    // rows 2 i and 2 i + 1
    __device__ __forceinline__ uint64_t pair(int i) const {
        if constexpr (FMT == DOSE_FMT_U16_SCALE) {
            // the codes under the exponent of 2^23 (byte permutations), minus 2^23
            return dev::f2_add(dev::f2_pack(__byte_perm(w[i], 0x4B00u, 0x5410u), __byte_perm(w[i], 0x4B00u, 0x5432u)),
                               dev::f2_splat(-8388608.0f));
        } else if constexpr (FMT == DOSE_FMT_BF16) {
            return dev::f2_pack(w[i] << 16, w[i] & 0xFFFF0000u);
        } else if constexpr (FMT == DOSE_FMT_F16) {
            return dev::f2_packf(dev::f16_to_f32((uint16_t)(w[i] & 0xFFFFu)), dev::f16_to_f32((uint16_t)(w[i] >> 16)));
        } else if constexpr (FMT == DOSE_FMT_F32) {
            return dev::f2_pack(w[2 * i], w[2 * i + 1]);
        } else {
            const uint32_t q = w[i >> 1];
            uint32_t h;
            asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h) : "h"((uint16_t)((i & 1) ? q >> 16 : q & 0xFFFFu)));
            return dev::f2_packf(dev::f16_to_f32((uint16_t)(h & 0xFFFFu)), dev::f16_to_f32((uint16_t)(h >> 16)));
        }
    }
};

template <uint32_t IW>
__device__ __forceinline__ uint32_t rg_col(const unsigned char* cols, uint32_t u) {
    return IW == 2 ? reinterpret_cast<const uint16_t*>(cols)[u] : reinterpret_cast<const uint32_t*>(cols)[u];
}

// ---- a packet in its slot
template <int FMT, int HR, uint32_t IW>
struct RgSlotView {
    uint32_t ng, nu;
    const uint32_t* gn;         // union columns of each group
    const uint32_t* rows;       // HR per group
    const float* scales;        // FP8: HR per group
    const unsigned char* cols;  // IW bytes each
    const unsigned char* vals;
    __device__ __forceinline__ explicit RgSlotView(const unsigned char* s) {
        const uint2 h = *reinterpret_cast<const uint2*>(s);
        ng = h.x;
        nu = h.y;
        gn = reinterpret_cast<const uint32_t*>(s) + 4;
        const unsigned char* p = s + 16 + ((4 * ng + 15) & ~15u);
        rows = reinterpret_cast<const uint32_t*>(p);
        p += 4 * HR * ng;
        scales = reinterpret_cast<const float*>(p);
        if (FMT == DOSE_FMT_FP8E4M3_ROWSCALE) p += 4 * HR * ng;
        cols = p;
        vals = p + ((nu * IW + 15) & ~15u);
    }
};

// Debug-checked builds (DOSE_DEBUG_CHECKS): whether a packet's parts lie inside
// its slot, its rows inside the matrix and its columns inside the CTA's list; a
// packet that does not is recorded (kErrBounds) and skipped by the whole warp.
template <int FMT, int HR, uint32_t IW>
__device__ __forceinline__ bool rg_packet_ok(const RgSlotView<FMT, HR, IW>& S, const unsigned char* slot, uint32_t cap,
                                             uint32_t nrows, uint32_t ncta, uint32_t lane, int* err) {
#ifdef DOSE_DEBUG_CHECKS
    bool ok = S.ng * HR <= kRgMaxRows && (uint32_t)(S.vals - slot) + S.nu * RgVal<FMT, HR>::kBytes <= cap;
    if (ok) {
        uint32_t sum = 0;
        for (uint32_t g = 0; g < S.ng; ++g) sum += S.gn[g];
        ok = sum == S.nu;
        for (uint32_t k = lane; k < S.ng * HR; k += 32) ok = ok && (S.rows[k] == 0xFFFFFFFFu || S.rows[k] < nrows);
        for (uint32_t k = lane; k < S.nu; k += 32) ok = ok && rg_col<IW>(S.cols, k) < ncta;
    }
    return dev::in_bounds(__all_sync(0xffffffffu, ok), err);
#else
    (void)S, (void)slot, (void)cap, (void)nrows, (void)ncta, (void)lane, (void)err;
    return true;
#endif
}

// ---- a warp's stream: its packets in order through its own ring.  Every lane
// keeps the same state; lane 0 issues the copies.  A packet is waited for, used
// by the whole warp, and its slot refilled (done()) with the packet `depth`
// further on.  NEED: packets without any of these flags are skipped.
template <uint32_t NEED>
struct RgStream {
    const uint4* pk;
    const unsigned char* data;
    unsigned char* slots;
    uint64_t* full;
    uint32_t* flags;
    uint32_t i, end, depth, stride;  // i: next packet to issue
    uint4 nxt;                       // its entry (loaded a packet ahead)
    uint32_t pending = 0;            // issued and not yet done
    uint32_t st = 0, ph = 0;         // slot and phase of the packet at hand
    uint32_t is = 0;                 // slot of the next issue

    // In three steps, so that the caller's own first loads overlap these: range()
    // loads where the warp's packets lie, entry() the first one's entry, start()
    // sets the ring up and issues the first copies.
    __device__ __forceinline__ void range(const RgView& v, uint32_t cta, uint32_t nw, uint32_t w) {
        pk = v.pk;
        data = v.data;
        const uint32_t* b = v.deal + (size_t)cta * nw + w;
        i = __ldg(b);
        end = __ldg(b + 1);
    }
    __device__ __forceinline__ void entry() {
        if (i < end) nxt = __ldg(pk + i);
    }
    __device__ __forceinline__ void start(uint32_t w, uint32_t d, uint32_t slot_bytes, unsigned char* smem,
                                          unsigned char* slot_base, uint32_t lane) {
        depth = d;
        stride = slot_bytes;
        full = reinterpret_cast<uint64_t*>(smem) + kRgMaxDepth * w;
        flags = reinterpret_cast<uint32_t*>(smem + 1024) + kRgMaxDepth * w;
        slots = slot_base + (size_t)w * d * slot_bytes;
        if (lane == 0) {
            for (uint32_t k = 0; k < d; ++k) dev::mbar_init(&full[k], 1);
            dev::fence_mbar_init();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
        fill(lane);
    }
    // First copies into an empty ring.
    __device__ __forceinline__ void fill(uint32_t lane) {
        is = st;
        for (uint32_t k = 0; k < depth; ++k) issue(lane);
    }
    __device__ __forceinline__ void issue(uint32_t lane) {
        if (i < end && !(nxt.y & NEED)) {
            do {
                ++i;
                if (i < end) nxt = __ldg(pk + i);
            } while (i < end && !(nxt.y & NEED));
        }
        if (i >= end) return;
        if (lane == 0) {
            const uint32_t bytes = (nxt.y & RG_SIZE_MASK) * 16;
            flags[is] = nxt.y;
            dev::mbar_arrive_expect_tx(&full[is], bytes);
            dev::bulk_g2s(slots + (size_t)is * stride, data + (uint64_t)nxt.x * 16, bytes, &full[is]);
        }
        ++pending;
        ++i;
        if (i < end) nxt = __ldg(pk + i);
        if (++is == depth) is = 0;
    }
    // Wait for the packet at hand; false on timeout (the copies in flight are then
    // waited for, with the same bound, before the warp gives up).
    __device__ __forceinline__ bool wait(int* err) {
        const bool ok = dev::mbar_wait_poll(&full[st], ph);
        if (__all_sync(0xffffffffu, ok)) {
            __syncwarp();  // lane 0's flag word is visible to every lane
            return true;
        }
        atomicExch(err, kErrTimeoutFull);
        while (pending) {
            dev::mbar_wait_poll(&full[st], ph);
            step();
        }
        return false;
    }
    __device__ __forceinline__ const unsigned char* slot() const { return slots + (size_t)st * stride; }
    __device__ __forceinline__ uint32_t flag() const { return flags[st]; }
    __device__ __forceinline__ void step() {
        --pending;
        if (++st == depth) {
            st = 0;
            ph ^= 1;
        }
    }
    __device__ __forceinline__ void done(uint32_t lane) {
        __syncwarp();  // every lane has read the slot
        step();
        issue(lane);
    }
};

// The row sums of a group over its union columns: acc[i] += values of rows
// 2 i, 2 i + 1 times x, lane l taking columns l, l + 32, ...  Up to four steps
// of 32 columns are loaded before the first product; only the last step of a
// call is masked (its lanes past n read nothing and add 0 * the zero element).
template <int FMT, int HR, uint32_t IW, int K>
__device__ __forceinline__ void rg_dot_steps(const unsigned char* cols, const unsigned char* vals, uint32_t n,
                                             uint32_t lane, const float* xs, uint32_t zc, uint64_t* acc) {
    RgVal<FMT, HR> q[K];
    uint32_t c[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t u = 32 * k + lane;
        if (k < K - 1 || u < n) {
            c[k] = rg_col<IW>(cols, u);
            q[k].load(vals + u * RgVal<FMT, HR>::kBytes);
        } else {
            c[k] = zc;
            q[k].zero();
        }
    }
    float x[K];
#pragma unroll
    for (int k = 0; k < K; ++k) x[k] = xs[c[k]];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint64_t xx = dev::f2_splat(x[k]);
#pragma unroll
        for (int i = 0; i < HR / 2; ++i) acc[i] = dev::f2_fma(q[k].pair(i), xx, acc[i]);
    }
}

template <int FMT, int HR, uint32_t IW>
__device__ __forceinline__ void rg_dot(const unsigned char* cols, const unsigned char* vals, uint32_t n, uint32_t lane,
                                       const float* xs, uint32_t zc, uint64_t* acc) {
    constexpr uint32_t VB = RgVal<FMT, HR>::kBytes;
    while (n > 128) {
        rg_dot_steps<FMT, HR, IW, 4>(cols, vals, 128, lane, xs, zc, acc);
        cols += 128 * IW;
        vals += 128 * VB;
        n -= 128;
    }
    switch ((n + 31) >> 5) {
        case 1: rg_dot_steps<FMT, HR, IW, 1>(cols, vals, n, lane, xs, zc, acc); break;
        case 2: rg_dot_steps<FMT, HR, IW, 2>(cols, vals, n, lane, xs, zc, acc); break;
        case 3: rg_dot_steps<FMT, HR, IW, 3>(cols, vals, n, lane, xs, zc, acc); break;
        default: rg_dot_steps<FMT, HR, IW, 4>(cols, vals, n, lane, xs, zc, acc); break;
    }
}

// Totals over the warp of HR row sums (a transposed butterfly): lane l returns
// row l / (32 / HR)'s total, the same value in all of that row's lanes.  Every
// sum is the same tree (l with l ^ 16, then ^ 8, ^ 4, ^ 2, ^ 1) for any HR.
template <int HR>
__device__ __forceinline__ float rg_reduce(const uint64_t (&acc)[HR / 2], uint32_t lane) {
    float a[HR];
#pragma unroll
    for (int i = 0; i < HR / 2; ++i) dev::f2_split(acc[i], a[2 * i], a[2 * i + 1]);
    uint32_t o = 16;
#pragma unroll
    for (int n = HR / 2; n >= 1; n /= 2, o /= 2) {
        const bool hi = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float keep = hi ? a[i + n] : a[i], send = hi ? a[i] : a[i + n];
            a[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, o));
        }
    }
    for (; o > 0; o /= 2) a[0] = __fadd_rn(a[0], __shfl_xor_sync(0xffffffffu, a[0], o));
    return a[0];
}

// The zeros the bulk stores read, written by the storing warp before any of them.
__device__ __forceinline__ void rg_fill_zeros(unsigned char* z, uint32_t lane) {
    for (uint32_t k = lane; k < kRgZeroBytes / 16; k += 32) reinterpret_cast<uint4*>(z)[k] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
}

// Rows without entries get zeros: one warp per CTA, a run per lane.  The
// 16-byte-aligned middle of a run goes out as bulk stores of a zeroed piece of
// shared memory (88 % of the clinical beam's rows are empty: 37 MB of dose that
// cost the warp a few instructions per 4 KB), the ends as words.
__device__ __forceinline__ void rg_zero_rows(const uint2* runs, uint32_t n, unsigned char* out, uint32_t row_bytes,
                                             const unsigned char* zeros, uint32_t lane) {
    for (uint32_t i = lane * gridDim.x + blockIdx.x; i < n; i += gridDim.x * 32) {  // (evenly over the CTAs first)
        const uint2 r = __ldg(runs + i);
        unsigned char* b = out + (uint64_t)r.x * row_bytes;
        unsigned char* e = b + (uint64_t)r.y * row_bytes;
        while (b < e && (reinterpret_cast<uintptr_t>(b) & 15u)) {
            *reinterpret_cast<uint32_t*>(b) = 0u;
            b += 4;
        }
        while (e > b && (reinterpret_cast<uintptr_t>(e) & 15u)) {
            e -= 4;
            *reinterpret_cast<uint32_t*>(e) = 0u;
        }
        while (b < e) {
            const uint32_t m = (uint32_t)min((unsigned long long)(e - b), (unsigned long long)kRgZeroBytes);
            dev::bulk_s2g(b, zeros, m);
            b += m;
        }
    }
    dev::bulk_store_wait();
}

#endif  // __CUDACC__

}  // namespace dose
