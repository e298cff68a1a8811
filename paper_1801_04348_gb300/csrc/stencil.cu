// The paper's two other parametric kernels (Section 5), with their own case
// discussion through the same walk as the GEMM (case_walk.cuh):
//
// Matrix transposition (Fig. "transpose"): c = a^T on 32-bit words.  A block of
// B0 x B1 threads owns B0 rows and B1*s columns of a; thread (u0, u1) handles
// columns u1 + k*B1, k < s (the paper's granularity s along j).
//   (4a,3a)  both a and c tile staged in shared memory, granularity s,
//   (3b,4a)  the same with s = 1,
//   (3b,4b)  no shared memory: each thread copies one word directly.
// (The figure prints c[i*N+j] = a[i][j], a copy; the kernel computes the
// transposition the text describes.)
//
// 1D Jacobi (Fig. "1dj"): int32 a[2N]; time step t writes one half from the
// three-point average of the other (t odd: a[p+1] = (a[N+p] + a[N+p+1] +
// a[N+p+2]) / 3, else a[N+p+1] = (a[p] + a[p+1] + a[p+2]) / 3) for every interior
// p in [0, N-2), integer division truncating toward zero.  A block of B threads
// owns s*B consecutive p, thread j handles p = p0 + j + k*B, k < s.
//   (4a,3a)  the read window (s*B + 2 words) and the s*B results are staged in
//            shared memory: 2 s B + 2 words, the figure's first case system,
//   (3b,4a)  the same with s = 1,
//   (3b,4b)  no shared memory.
// One launch per time step (the halves swap roles between steps).
#include <cooperative_groups.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "case_walk.cuh"
#include "pgk_internal.cuh"

namespace pgk {

struct TArgs {
    int rows, cols;
    const uint32_t* src;
    int lds;
    uint32_t* dst;
    int ldd;
};

// ------------------------------------------------------------ transposition
template <int S>
__global__ void k_transpose_cached(TArgs p) {
    extern __shared__ uint32_t tile_t[];  // B0 x (B1 S + 1)
    const int B0 = blockDim.y, B1 = blockDim.x;
    const int W = B1 * S, P = W + 1;
    const int tiles_n = (p.cols + W - 1) / W;
    const int r0 = (blockIdx.x / tiles_n) * B0, c0 = (blockIdx.x % tiles_n) * W;
    const int u0 = threadIdx.y, u1 = threadIdx.x;
    const int gi = r0 + u0;
#pragma unroll
    for (int k = 0; k < S; ++k) {
        const int j = u1 + k * B1;
        const int gj = c0 + j;
        tile_t[u0 * P + j] = (gi < p.rows && gj < p.cols) ? __ldg(p.src + (size_t)gi * p.lds + gj) : 0u;
    }
    __syncthreads();
    // output row c0 + j holds elements r0 .. r0 + B0 - 1: consecutive threads write
    // consecutive elements of one output row.  Thread t writes element i = t mod B0
    // of output rows j = t div B0 + m B1 (m = 0 .. S - 1): one division per thread
    const int tid = u0 * B1 + u1;
    const int i = tid % B0, j0 = tid / B0;
    if (r0 + i < p.rows) {
#pragma unroll
        for (int m = 0; m < S; ++m) {
            const int j = j0 + m * B1;
            if (c0 + j < p.cols) p.dst[(size_t)(c0 + j) * p.ldd + r0 + i] = tile_t[i * P + j];
        }
    }
}

__global__ void k_transpose_direct(TArgs p) {
    const int B0 = blockDim.y, B1 = blockDim.x;
    const int tiles_n = (p.cols + B1 - 1) / B1;
    const int i = (blockIdx.x / tiles_n) * B0 + threadIdx.y;
    const int j = (blockIdx.x % tiles_n) * B1 + threadIdx.x;
    if (i < p.rows && j < p.cols) p.dst[(size_t)j * p.ldd + i] = __ldg(p.src + (size_t)i * p.lds + j);
}

// The transposition without explicit parameters: a 64 x 64 tile per block, staged in
// shared memory with a pitch of 65 words.  Bound by HBM: a block reads 256-byte segments
// of source rows and writes 256-byte segments of destination rows, every thread with all
// of its 64 (VEC) or 32 bytes in flight before the barrier.  VEC moves 16 bytes per access
// (256 threads); otherwise 4 bytes per access and 512 threads, for bases or row strides
// that are not multiples of 16 bytes.  At order 2^14 on GB300 the (8, 32, 2) block that
// this replaces as the default takes 660 us (its 8-row tile writes 32-byte segments), VEC
// 312 us = 6.9 TB/s and the scalar form 326 us (256 threads: 347), against 323 us for a
// plain copy of the same bytes; tiles of 32 or 128 words a side, other walks over the
// tiles and streaming hints lie within 4 % of VEC.
template <bool VEC>
__global__ void __launch_bounds__(VEC ? 256 : 512) k_transpose_tile(TArgs p) {
    constexpr int T = 64, NT = VEC ? 256 : 512;
    __shared__ uint32_t t[T][T + 1];
    const int tiles_n = (p.cols + T - 1) / T;
    const int r0 = (int)(blockIdx.x / tiles_n) * T, c0 = (int)(blockIdx.x % tiles_n) * T;
    const int tid = threadIdx.x;
    if (VEC) {
        constexpr int L = T * T / 4 / NT, Q = T / 4;
        uint4 v[L];
#pragma unroll
        for (int i = 0; i < L; ++i) {
            const int r = (tid + i * NT) / Q, c = (tid + i * NT) % Q * 4;
            v[i] = make_uint4(0u, 0u, 0u, 0u);
            if (r0 + r < p.rows) {
                const uint32_t* s = p.src + (size_t)(r0 + r) * p.lds + c0 + c;
                const int n = p.cols - c0 - c;
                if (n >= 4) {
                    v[i] = __ldg(reinterpret_cast<const uint4*>(s));
                } else {
                    if (n > 0) v[i].x = __ldg(s);
                    if (n > 1) v[i].y = __ldg(s + 1);
                    if (n > 2) v[i].z = __ldg(s + 2);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < L; ++i) {
            uint32_t* d = &t[(tid + i * NT) / Q][(tid + i * NT) % Q * 4];
            d[0] = v[i].x;
            d[1] = v[i].y;
            d[2] = v[i].z;
            d[3] = v[i].w;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < L; ++i) {
            const int j = (tid + i * NT) / Q, r = (tid + i * NT) % Q * 4;
            if (c0 + j >= p.cols) continue;
            uint32_t* d = p.dst + (size_t)(c0 + j) * p.ldd + r0 + r;
            const int n = p.rows - r0 - r;
            if (n >= 4) {
                *reinterpret_cast<uint4*>(d) = make_uint4(t[r][j], t[r + 1][j], t[r + 2][j], t[r + 3][j]);
            } else {
                if (n > 0) d[0] = t[r][j];
                if (n > 1) d[1] = t[r + 1][j];
                if (n > 2) d[2] = t[r + 2][j];
            }
        }
    } else {
        constexpr int L = T * T / NT;
        uint32_t v[L];
#pragma unroll
        for (int i = 0; i < L; ++i) {
            const int r = r0 + (tid + i * NT) / T, c = c0 + (tid + i * NT) % T;
            v[i] = (r < p.rows && c < p.cols) ? __ldg(p.src + (size_t)r * p.lds + c) : 0u;
        }
#pragma unroll
        for (int i = 0; i < L; ++i) t[(tid + i * NT) / T][(tid + i * NT) % T] = v[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < L; ++i) {
            const int j = (tid + i * NT) / T, r = (tid + i * NT) % T;
            if (c0 + j < p.cols && r0 + r < p.rows) p.dst[(size_t)(c0 + j) * p.ldd + r0 + r] = t[r][j];
        }
    }
}

static cudaError_t launch_transpose_tile(const TArgs& a, cudaStream_t st) {
    const long long tiles = (long long)((a.rows + 63) / 64) * ((a.cols + 63) / 64);
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    // 16-byte accesses need both bases and both row strides on 16-byte boundaries
    const bool vec = ((uintptr_t)a.src & 15u) == 0 && ((uintptr_t)a.dst & 15u) == 0 && a.lds % 4 == 0 &&
                     a.ldd % 4 == 0;
    if (vec)
        k_transpose_tile<true><<<(unsigned)tiles, 256, 0, st>>>(a);
    else
        k_transpose_tile<false><<<(unsigned)tiles, 512, 0, st>>>(a);
    return cudaGetLastError();
}

template <int S>
static cudaError_t launch_transpose_cached(const TArgs& a, int B0, int B1, int smem, cudaStream_t st) {
    const long long tiles = (long long)((a.rows + B0 - 1) / B0) * ((a.cols + B1 * S - 1) / (B1 * S));
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute((const void*)k_transpose_cached<S>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    k_transpose_cached<S><<<(unsigned)tiles, dim3(B1, B0), smem, st>>>(a);
    return cudaGetLastError();
}

static cudaError_t launch_transpose_direct(const TArgs& a, int B0, int B1, int, cudaStream_t st) {
    const long long tiles = (long long)((a.rows + B0 - 1) / B0) * ((a.cols + B1 - 1) / B1);
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    k_transpose_direct<<<(unsigned)tiles, dim3(B1, B0), 0, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- 1D Jacobi
template <int S>
__global__ void k_jacobi_cached(int n, int odd, int32_t* a) {
    extern __shared__ int32_t win_j[];  // read window (S B + 2) then results (S B)
    const int B = blockDim.x, j = threadIdx.x;
    const int p0 = blockIdx.x * S * B;
    const int32_t* src = odd ? a + n : a;
    int32_t* dst = odd ? a : a + n;
    int32_t* out = win_j + S * B + 2;
    for (int idx = j; idx < S * B + 2; idx += B) win_j[idx] = (p0 + idx < n) ? src[p0 + idx] : 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < S; ++k) {
        const int q = j + k * B;
        out[q] = (win_j[q] + win_j[q + 1] + win_j[q + 2]) / 3;
    }
#pragma unroll
    for (int k = 0; k < S; ++k) {
        const int q = j + k * B, pp = p0 + q;
        if (pp < n - 2) dst[pp + 1] = out[q];
    }
}

__global__ void k_jacobi_direct(int n, int odd, int32_t* a) {
    const int pp = blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t* src = odd ? a + n : a;
    int32_t* dst = odd ? a : a + n;
    if (pp < n - 2) dst[pp + 1] = (src[pp] + src[pp + 1] + src[pp + 2]) / 3;
}

// Several time steps in one cooperative launch, for calls without parameters whose array the
// blocks can hold: block b keeps interior points [1 + b R, 1 + (b + 1) R) in shared memory
// with a halo of up to JSTEPS points a side, and recomputes the halo instead of exchanging
// it.  A group of up to JSTEPS steps reads its window from the first half, waits until every
// block has read (the group overwrites both halves), takes the steps, and writes the results
// of the last two, which are what the halves then hold.  The end points of each half never
// change.  A launch per step pays 4.1 us each, and at the paper's length 2^15 + 2 the work
// of a step is far below that: 4 steps take 6.1 us instead of 16.4, at 2^20 + 2 points 10.4
// instead of 24.7 (20.4 with granularity 8).
static constexpr int JSTEPS = 8;   // even: every group starts from the first half
static constexpr int JTHREADS = 512;

__global__ void __launch_bounds__(JTHREADS, 2) k_jacobi_steps(int n, int steps, int R, int32_t* a) {
    extern __shared__ int32_t buf_j[];   // two windows of R + 2 JSTEPS points
    const int lo = 1 + (int)min((long long)blockIdx.x * R, (long long)(n - 2));
    const int hi = lo + min(R, n - 1 - lo);   // own points [lo, hi)
    int32_t* cur = buf_j;
    int32_t* nxt = buf_j + R + 2 * JSTEPS;
    for (int t0 = 0; t0 < steps; t0 += JSTEPS) {
        const int s = min(JSTEPS, steps - t0);
        const int w0 = max(0, lo - s), w1 = min(n, hi + s);   // window [w0, w1)
        for (int i = w0 + (int)threadIdx.x; i < w1; i += JTHREADS) cur[i - w0] = a[i];
        // end points of the second half (those of the first lie in the windows that need them)
        const int32_t b0 = a[n], b1 = a[2 * (size_t)n - 1], c0 = a[0], c1 = a[n - 1];
        if (s > 1) cooperative_groups::this_grid().sync();
        else __syncthreads();
        for (int k = 1; k <= s; ++k) {
            const bool odd = k & 1;   // step t0 + k - 1 is even and writes the second half
            int32_t* half = odd ? a + n : a;
            const int p0 = max(0, lo - (s - k)), p1 = min(n, hi + (s - k));
            for (int i = p0 + (int)threadIdx.x; i < p1; i += JTHREADS) {
                const int j = i - w0;
                int32_t v;
                if (i == 0) v = odd ? b0 : c0;
                else if (i == n - 1) v = odd ? b1 : c1;
                else v = (cur[j - 1] + cur[j] + cur[j + 1]) / 3;
                nxt[j] = v;
                if (k >= s - 1 && i >= lo && i < hi) half[i] = v;
            }
            __syncthreads();
            int32_t* const t = cur;
            cur = nxt;
            nxt = t;
        }
        if (t0 + JSTEPS < steps) cooperative_groups::this_grid().sync();
    }
}

// Launches k_jacobi_steps; false if it does not apply (one step, an array too long for the
// blocks' shared memory, a stream being captured, blocks that cannot all be resident): the
// caller then launches every step.
static bool launch_jacobi_steps(int n, int steps, int32_t* a, cudaStream_t st, cudaError_t* err) {
    pgk_machine m;
    if (steps < 2 || current_machine(&m, NULL) != PGK_OK) return false;
    // at least JTHREADS points per block, two blocks per SM, their windows within 100 KB
    const int blocks = (int)std::min<long long>(((long long)n - 2 + JTHREADS - 1) / JTHREADS, 2LL * m.sm_count);
    const long long R = ((long long)n - 2 + blocks - 1) / blocks;
    const long long smem = 8 * (R + 2 * JSTEPS);
    if (smem > 100 * 1024 || 2 * (smem + 1024) > 227 * 1024) return false;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    static SmemLimit limit;
    if (allow_smem(limit, (const void*)k_jacobi_steps, 100 * 1024) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks, 1, 1);
    cfg.blockDim = dim3(JTHREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    *err = cudaLaunchKernelEx(&cfg, k_jacobi_steps, n, steps, (int)R, a);
    if (*err == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        return false;
    }
    return true;
}

// ----------------------------------------------------------- variant tables
enum { KIND_TRANSPOSE = 0, KIND_JACOBI = 1 };

struct StencilVariant {
    int kind, cached, s;
    const void* func;
};

static const StencilVariant* stencil_table(int* n) {
    static const StencilVariant t[] = {
        {KIND_TRANSPOSE, 1, 1, (const void*)k_transpose_cached<1>},
        {KIND_TRANSPOSE, 1, 2, (const void*)k_transpose_cached<2>},
        {KIND_TRANSPOSE, 1, 4, (const void*)k_transpose_cached<4>},
        {KIND_TRANSPOSE, 1, 8, (const void*)k_transpose_cached<8>},
        {KIND_TRANSPOSE, 0, 1, (const void*)k_transpose_direct},
        {KIND_JACOBI, 1, 1, (const void*)k_jacobi_cached<1>},
        {KIND_JACOBI, 1, 2, (const void*)k_jacobi_cached<2>},
        {KIND_JACOBI, 1, 4, (const void*)k_jacobi_cached<4>},
        {KIND_JACOBI, 1, 8, (const void*)k_jacobi_cached<8>},
        {KIND_JACOBI, 0, 1, (const void*)k_jacobi_direct},
    };
    *n = (int)(sizeof(t) / sizeof(t[0]));
    return t;
}

static int stencil_base_id = -1;

void register_stencil_variants(std::vector<Variant>& v) {
    int n;
    const StencilVariant* t = stencil_table(&n);
    stencil_base_id = (int)v.size();
    for (int i = 0; i < n; ++i) {
        Variant x;
        memset(&x.info, 0, sizeof(x.info));
        x.info.family = t[i].kind == KIND_TRANSPOSE
                            ? (t[i].cached ? PGK_FAM_TRANSPOSE : PGK_FAM_TRANSPOSE_DIRECT)
                            : (t[i].cached ? PGK_FAM_JACOBI : PGK_FAM_JACOBI_DIRECT);
        x.info.s = t[i].s;
        x.info.sr = 1;
        x.info.regs = -1;
        x.info.max_threads = -1;
        x.func = t[i].func;
        x.launch = nullptr;
        x.smem_fixed = 0;
        v.push_back(x);
    }
}

static int stencil_variant(int kind, int cached, int s) {
    registry();
    int n;
    const StencilVariant* t = stencil_table(&n);
    for (int i = 0; i < n; ++i)
        if (t[i].kind == kind && t[i].cached == cached && (!cached || t[i].s == s))
            return stencil_base_id + i;
    return -1;
}

// Register classes of a caller-supplied table (5 entries): cached s = 1, 2, 4, 8; direct.
static int stencil_reg_class(int cached, int s) {
    if (!cached) return 4;
    return s == 1 ? 0 : s == 2 ? 1 : s == 4 ? 2 : 3;
}

// Program state and evaluation functions of the transposition / Jacobi family
// for walk_cases.  There is no register-capped build: strategy "1" leaves the
// register count unchanged, so a refused register counter stays refused.
struct StencilSpec {
    struct Prog {
        int cache, s, gran, regopt;
    };
    int kind;
    int threads;      // B0 * B1 (transposition) or B (Jacobi)
    int B0, B1;       // transposition tile rows / thread columns
    const int* table; // caller register table or NULL

    long long smem(const Prog& p) const {
        if (!p.cache) return 0;
        if (kind == KIND_TRANSPOSE) return 4LL * B0 * ((long long)B1 * p.s + 1);
        return 4LL * (2LL * p.s * threads + 2);  // 2 s B + 2 words (Fig. "1dj")
    }

    pgk_status regs(const Prog& p, long long* out) const {
        if (table) {
            *out = table[stencil_reg_class(p.cache, p.s)];
            return PGK_OK;
        }
        const int id = stencil_variant(kind, p.cache, p.s);
        if (id < 0) {
            set_error("no compiled variant for s=%d", p.s);
            return PGK_ERR_UNSUPPORTED;
        }
        int r = -1;
        pgk_status st = variant_attrs(id, &r, NULL);
        if (st != PGK_OK) return st;
        *out = r;
        return PGK_OK;
    }

    pgk_status eval(int c, const Prog& p, long long* v) const {
        switch (c) {
            case C_THREADS: *v = threads; return PGK_OK;
            case C_REGS: return regs(p, v);
            case C_REGALLOC: {
                long long r = 0;
                pgk_status st = regs(p, &r);
                if (st != PGK_OK) return st;
                *v = regalloc_bytes(threads, r);
                return PGK_OK;
            }
            default: *v = smem(p); return PGK_OK;
        }
    }

    void apply(int o, Prog& p) const {
        if (o == O_REG) p.regopt = 1;
        else if (o == O_GRAN) { p.s = 1; p.gran = 1; }
        else p.cache = 0;
    }
};

static pgk_status stencil_case(int kind, const pgk_machine* m, const int* table, const pgk_params* prog,
                               pgk_case* out) {
    if (!m || !prog || !out) {
        set_error("NULL argument");
        return PGK_ERR_INVALID_ARG;
    }
    const int s = prog->s;
    const int B0 = prog->B0, B1 = kind == KIND_TRANSPOSE ? prog->B1 : 1;
    if (B0 < 1 || B1 < 1 || s < 1 || B0 > 4096 || B1 > 4096) {
        set_error("program parameters must be positive (B0=%d B1=%d s=%d)", B0, B1, s);
        return PGK_ERR_INVALID_ARG;
    }
    if (!(s == 1 || s == 2 || s == 4 || s == 8)) {
        set_error("variants exist for s in {1,2,4,8}, got %d", s);
        return PGK_ERR_UNSUPPORTED;
    }
    StencilSpec spec;
    spec.kind = kind;
    spec.threads = B0 * B1;
    spec.B0 = B0;
    spec.B1 = B1;
    spec.table = table;
    StencilSpec::Prog p = {1, s, 0, 0};
    pgk_status st = walk_cases(*m, spec, p);
    if (st != PGK_OK) return st;
    pgk_case cs;
    memset(&cs, 0, sizeof(cs));
    cs.leaf = !p.cache ? PGK_LEAF_3B4B : (p.gran ? PGK_LEAF_3B4A : PGK_LEAF_4A3A);
    cs.family = kind == KIND_TRANSPOSE ? (p.cache ? PGK_FAM_TRANSPOSE : PGK_FAM_TRANSPOSE_DIRECT)
                                       : (p.cache ? PGK_FAM_JACOBI : PGK_FAM_JACOBI_DIRECT);
    cs.regopt = p.regopt;
    cs.variant_id = stencil_variant(kind, p.cache, p.s);
    long long r = 0;
    spec.eval(C_REGS, p, &r);
    cs.regs = (int)r;
    cs.smem_bytes = (int)spec.smem(p);
    cs.threads = spec.threads;
    cs.params.B0 = B0;
    cs.params.B1 = B1;
    cs.params.s = p.cache ? p.s : 1;
    cs.params.sr = 1;
    cs.params.tile = 0;
    *out = cs;
    return PGK_OK;
}

static pgk_status run_transpose(const pgk_case& c, int rows, int cols, const void* src, int lds,
                                void* dst, int ldd, cudaStream_t st) {
    TArgs a = {rows, cols, (const uint32_t*)src, lds, (uint32_t*)dst, ldd};
    const int B0 = c.params.B0, B1 = c.params.B1;
    cudaError_t e;
    if (c.family == PGK_FAM_TRANSPOSE_DIRECT) {
        e = launch_transpose_direct(a, B0, B1, 0, st);
    } else if (c.family == PGK_FAM_TRANSPOSE) {
        switch (c.params.s) {
            case 1: e = launch_transpose_cached<1>(a, B0, B1, c.smem_bytes, st); break;
            case 2: e = launch_transpose_cached<2>(a, B0, B1, c.smem_bytes, st); break;
            case 4: e = launch_transpose_cached<4>(a, B0, B1, c.smem_bytes, st); break;
            default: e = launch_transpose_cached<8>(a, B0, B1, c.smem_bytes, st); break;
        }
    } else {
        set_error("case is not a transposition case");
        return PGK_ERR_INVALID_ARG;
    }
    if (e != cudaSuccess) return cuda_fail(e, "transposition launch");
    return PGK_OK;
}

template <int S>
static cudaError_t launch_jacobi_cached(int n, int odd, int32_t* a, int B, int smem, cudaStream_t st) {
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute((const void*)k_jacobi_cached<S>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    const long long blocks = ((long long)n - 2 + (long long)S * B - 1) / ((long long)S * B);
    k_jacobi_cached<S><<<(unsigned)std::max(1LL, blocks), B, smem, st>>>(n, odd, a);
    return cudaGetLastError();
}

static pgk_status run_jacobi(const pgk_case& c, int n, int steps, int32_t* a, cudaStream_t st) {
    const int B = c.params.B0;
    for (int t = 0; t < steps; ++t) {
        const int odd = t & 1;
        cudaError_t e;
        if (c.family == PGK_FAM_JACOBI_DIRECT) {
            const long long blocks = ((long long)n - 2 + B - 1) / B;
            k_jacobi_direct<<<(unsigned)std::max(1LL, blocks), B, 0, st>>>(n, odd, a);
            e = cudaGetLastError();
        } else if (c.family == PGK_FAM_JACOBI) {
            switch (c.params.s) {
                case 1: e = launch_jacobi_cached<1>(n, odd, a, B, c.smem_bytes, st); break;
                case 2: e = launch_jacobi_cached<2>(n, odd, a, B, c.smem_bytes, st); break;
                case 4: e = launch_jacobi_cached<4>(n, odd, a, B, c.smem_bytes, st); break;
                default: e = launch_jacobi_cached<8>(n, odd, a, B, c.smem_bytes, st); break;
            }
        } else {
            set_error("case is not a Jacobi case");
            return PGK_ERR_INVALID_ARG;
        }
        if (e != cudaSuccess) return cuda_fail(e, "Jacobi launch");
    }
    return PGK_OK;
}

}  // namespace pgk

using namespace pgk;

extern "C" {

pgk_status pgk_select_case_transpose(const pgk_machine* machine, const int* regs_by_class, int rows,
                                     int cols, const pgk_params* prog, pgk_case* out) {
    if (rows < 1 || cols < 1) {
        set_error("sizes must be >= 1");
        return PGK_ERR_INVALID_ARG;
    }
    return stencil_case(KIND_TRANSPOSE, machine, regs_by_class, prog, out);
}

pgk_status pgk_transpose_case(const pgk_case* c, int rows, int cols, const void* src, int lds,
                              void* dst, int ldd, void* stream) {
    if (!c || rows < 1 || cols < 1 || !src || !dst || lds < cols || ldd < rows) {
        set_error("bad transposition arguments");
        return PGK_ERR_INVALID_ARG;
    }
    return run_transpose(*c, rows, cols, src, lds, dst, ldd, (cudaStream_t)stream);
}

pgk_status pgk_transpose(int rows, int cols, const void* src, int lds, void* dst, int ldd,
                         const pgk_params* prog, void* stream) {
    if (rows < 1 || cols < 1 || !src || !dst || lds < cols || ldd < rows) {
        set_error("bad transposition arguments");
        return PGK_ERR_INVALID_ARG;
    }
    if (!prog) {
        const TArgs a = {rows, cols, (const uint32_t*)src, lds, (uint32_t*)dst, ldd};
        const cudaError_t e = launch_transpose_tile(a, (cudaStream_t)stream);
        return e == cudaSuccess ? PGK_OK : cuda_fail(e, "transposition launch");
    }
    pgk_machine m;
    pgk_status st = current_machine(&m, NULL);
    if (st != PGK_OK) return st;
    pgk_case c;
    if ((st = stencil_case(KIND_TRANSPOSE, &m, NULL, prog, &c)) != PGK_OK) return st;
    return run_transpose(c, rows, cols, src, lds, dst, ldd, (cudaStream_t)stream);
}

pgk_status pgk_select_case_jacobi(const pgk_machine* machine, const int* regs_by_class, int n,
                                  const pgk_params* prog, pgk_case* out) {
    if (n < 3) {
        set_error("Jacobi needs n >= 3");
        return PGK_ERR_INVALID_ARG;
    }
    return stencil_case(KIND_JACOBI, machine, regs_by_class, prog, out);
}

pgk_status pgk_jacobi_case(const pgk_case* c, int n, int steps, int32_t* a, void* stream) {
    if (!c || n < 3 || steps < 0 || !a) {
        set_error("bad Jacobi arguments");
        return PGK_ERR_INVALID_ARG;
    }
    return run_jacobi(*c, n, steps, a, (cudaStream_t)stream);
}

pgk_status pgk_jacobi(int n, int steps, int32_t* a, const pgk_params* prog, void* stream) {
    if (n < 3 || steps < 0 || !a) {
        set_error("bad Jacobi arguments");
        return PGK_ERR_INVALID_ARG;
    }
    pgk_machine m;
    pgk_status st = current_machine(&m, NULL);
    if (st != PGK_OK) return st;
    // without parameters: the steps of one launch where the blocks can hold the array, else a
    // launch per step at the paper's best block (128, granularity 2: Table Jacobi), with
    // granularity 8 from 2^20 points on, where HBM and not the launch bounds a step
    // (4 steps at 2^26 points: 393 us, 788 with granularity 2)
    cudaError_t e = cudaSuccess;
    if (!prog && launch_jacobi_steps(n, steps, a, (cudaStream_t)stream, &e))
        return e == cudaSuccess ? PGK_OK : cuda_fail(e, "Jacobi launch");
    pgk_params p = {128, 1, n >= (1 << 20) ? 8 : 2, 1, 0};
    if (prog) p = *prog;
    pgk_case c;
    if ((st = stencil_case(KIND_JACOBI, &m, NULL, &p, &c)) != PGK_OK) return st;
    return run_jacobi(c, n, steps, a, (cudaStream_t)stream);
}

}  // extern "C"
