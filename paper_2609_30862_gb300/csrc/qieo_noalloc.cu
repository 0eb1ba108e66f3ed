// qieo_noalloc.cu -- qieo_generation_noalloc: one QIEO generation on caller-owned device
// buffers, with the library's working memory in a fixed device array instead of an
// allocation.
//
// Some callers cannot call cudaMalloc at the point where they need a generation: code
// running while a memory pool is locked or being torn down, real-time loops where an
// allocation may stall, and hosts whose allocator owns every byte of device memory. They
// hold their own input and output buffers; this entry point needs nothing else from
// them. Its per-row sums and block counter live in g_noalloc_scratch below,
// a file-scope __device__ array of kNoallocScratchBytes that every GPU which loads the
// library keeps until the process exits.
//
// The host never dereferences g_noalloc_scratch: in host code that name is only a
// stand-in for the device symbol. The device address is looked up once per device with
// cudaGetSymbolAddress (with that device current) on the first call made on it, and is
// passed to the kernels. Device code reaches the array only through that pointer.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdarg>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/qieo.h"
#include "qieo_device.cuh"

namespace qieo_internal {
void set_last_error(const char *msg);   // defined with qieo_last_error() in qieo_api.cu
}

namespace {

constexpr int kThreads = 256;
constexpr int kMaxD = 4000;
constexpr int kMaxThr = kMaxD / 2 + 1;

// Scratch layout: [0, 256) block counter; [256, 256 + 16 * kNoallocMaxNp) row sums
// (int64 weight sum, int64 value sum per chromosome).
constexpr size_t kCounterBytes = 256;
constexpr size_t kNoallocScratchBytes = kCounterBytes + 16 * (size_t)QIEO_NOALLOC_MAX_NP;

__device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
unsigned char *g_scratch_ptr[kMaxDevices];     // device address of g_noalloc_scratch

qieo_status noalloc_fail(qieo_status st, const char *fmt, ...) __attribute__((format(printf, 2, 3)));
qieo_status noalloc_fail(qieo_status st, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    qieo_internal::set_last_error(buf);   // read back through qieo_last_error()
    return st;
}

// Observation thresholds passed by value (kernel parameter space), so the call needs no
// copy into device memory either. Two sizes, so that the usual step counts (D <= 508) do not
// send 8 KB of parameters with every launch.
constexpr int kSmallThr = 255;

template <int kThr>
struct NoallocArgs {
    const int32_t *w, *v;
    int16_t *k;
    uint8_t *x;
    int64_t *fitness;
    int32_t *elite;
    unsigned int *counter;
    long long *sums;              // [2 np]
    int64_t capacity, lambda;
    int32_t ng, np, K;
    int32_t t;
    int32_t ntile, rows;          // tiles of kTileGenes genes per row; rows per warp
    uint32_t seed, inst;
    uint32_t thr[kThr];           // low 32 bits of T[n]; T[2K] = 2^32 is handled as "always 1"
};

__device__ __forceinline__ void grid_dependency_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void allow_dependent_launch()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__global__ void __launch_bounds__(kThreads) noalloc_clear_kernel(unsigned int *counter,
                                                                 long long *sums, int32_t n)
{
    allow_dependent_launch();
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i == 0) *counter = 0u;
    for (int j = i; j < n; j += gridDim.x * kThreads) sums[j] = 0;
}

// Eight consecutive halfwords at p + i (i + 8 <= total) as four words, from at most two
// aligned 16-byte loads that lie inside p[0 .. total); element loads at the buffer's ends.
__device__ __forceinline__ uint4 load_half8(const int16_t *p, size_t i, size_t total)
{
    const uintptr_t addr = reinterpret_cast<uintptr_t>(p + i), a0 = addr & ~(uintptr_t)15;
    const uint32_t m = (uint32_t)(addr & 15u);              // bytes past the aligned chunk
    uint32_t q[8];
    if (a0 >= reinterpret_cast<uintptr_t>(p) && a0 + (m ? 32 : 16) <= reinterpret_cast<uintptr_t>(p + total)) {
        const uint4 a = *reinterpret_cast<const uint4 *>(a0);
        if (m == 0u) return a;
        const uint4 b = *reinterpret_cast<const uint4 *>(a0 + 16);
        q[0] = a.x; q[1] = a.y; q[2] = a.z; q[3] = a.w;
        q[4] = b.x; q[5] = b.y; q[6] = b.z; q[7] = b.w;
        if (m & 8u) {
#pragma unroll
            for (int k = 0; k < 6; ++k) q[k] = q[k + 2];
        }
        if (m & 4u) {
#pragma unroll
            for (int k = 0; k < 5; ++k) q[k] = q[k + 1];
        }
        if (m & 2u) {
#pragma unroll
            for (int k = 0; k < 4; ++k) q[k] = __funnelshift_r(q[k], q[k + 1], 16);
        }
    } else {
        const uint16_t *h = reinterpret_cast<const uint16_t *>(p + i);
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = (uint32_t)h[2 * k] | ((uint32_t)h[2 * k + 1] << 16);
    }
    return make_uint4(q[0], q[1], q[2], q[3]);
}

// Eight consecutive bytes at p + i (i + 8 <= total), likewise.
__device__ __forceinline__ uint2 load_byte8(const uint8_t *p, size_t i, size_t total)
{
    const uintptr_t addr = reinterpret_cast<uintptr_t>(p + i), a0 = addr & ~(uintptr_t)7;
    const uint32_t m = (uint32_t)(addr & 7u);
    if (a0 >= reinterpret_cast<uintptr_t>(p) && a0 + (m ? 16 : 8) <= reinterpret_cast<uintptr_t>(p + total)) {
        uint2 a = *reinterpret_cast<const uint2 *>(a0);
        if (m == 0u) return a;
        const uint2 b = *reinterpret_cast<const uint2 *>(a0 + 8);
        uint32_t q0 = a.x, q1 = a.y, q2 = b.x;
        if (m & 4u) {
            q0 = a.y;
            q1 = b.x;
            q2 = b.y;
        }
        const uint32_t sh = 8u * (m & 3u);
        return make_uint2(__funnelshift_r(q0, q1, sh), __funnelshift_r(q1, q2, sh));
    }
    uint32_t r[2] = {0u, 0u};
#pragma unroll
    for (int k = 0; k < 8; ++k) r[k >> 2] |= (uint32_t)p[i + k] << (8 * (k & 3));
    return make_uint2(r[0], r[1]);
}

// Sum over the warp of a 64-bit value of at most 36 bits and a sign, as two 32-bit
// reductions: 21 low bits (32 of them stay below 2^26) and the signed rest.
__device__ __forceinline__ long long warp_sum(long long s)
{
    const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)s & 0x1fffffu);
    const int32_t hi = __reduce_add_sync(0xffffffffu, (int32_t)(s >> 21));
    return ((long long)hi << 21) + (long long)lo;
}

// Observation and the per-chromosome sums of generation t on the caller's int16 angle
// indices, then (last block) the penalised fitness and the lowest-index elite.
//
// A warp takes one tile of 256 genes and a.rows consecutive chromosomes: a lane keeps its
// 8 genes' items in registers over the rows, and a row costs one 16-byte read of its angle
// indices (two where the row is not 16-byte aligned; rows of the caller's buffers start at
// any even address), two Philox calls, one 8-byte store of its alleles and, per warp, one
// pair of 64-bit atomics. Rows of any alignment store whole aligned 8-byte words: a row's
// bytes are shifted by its misalignment with the neighbouring lane's, and only the first and
// the last lane of the tile store partial words. A thread per 8 genes with element accesses
// and two atomics each, which this replaces, spent its time on 1.3 M contended atomics and
// on single-byte stores (512 x 10,007 genes, a whole call with its rotation: 170 us, now 27 us, 19 of
// them in this kernel).
constexpr int kTileGenes = 256;

template <int kThr>
__global__ void __launch_bounds__(kThreads, 3) noalloc_observe_kernel(const __grid_constant__ NoallocArgs<kThr> a)
{
    __shared__ uint32_t s_thr[kThr];
    __shared__ int s_last;
    __shared__ int64_t s_f[kThreads / 32];
    __shared__ int32_t s_c[kThreads / 32];
    for (int i = threadIdx.x; i < 2 * a.K + 1; i += kThreads) s_thr[i] = a.thr[i];
    grid_dependency_wait();       // the sums are clear, the caller's earlier work is done
    __syncthreads();
    const unsigned char *thr_bytes = reinterpret_cast<const unsigned char *>(s_thr);

    const int lane = threadIdx.x & 31;
    const int64_t item = (int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    const int32_t tile = (int32_t)(item % a.ntile);
    const int64_t c_begin = item / a.ntile * a.rows;
    const int32_t c_end = (int32_t)min((int64_t)a.np, c_begin + a.rows);
    const size_t j0 = (size_t)tile * kTileGenes + 8u * lane;          // this lane's first gene
    const int32_t left = (int32_t)((int64_t)a.ng - (int64_t)j0);      // genes from there on
    const int32_t nv = min(8, left);                                  // its genes (<= 0: none)
    const size_t total = (size_t)a.np * a.ng;
    const uint32_t kk = (uint32_t)a.K * 0x00010001u, kneg = __vneg2(kk), off_top = 8u * (uint32_t)a.K;

    if (c_begin < a.np) {
        int32_t w[8], v[8];
        uint32_t any = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            w[i] = i < nv ? a.w[j0 + i] : 0;
            v[i] = i < nv ? a.v[j0 + i] : 0;
            any |= (uint32_t)w[i] | (uint32_t)v[i];
        }
        // Items below 2^8: a lane's 8 alleles and both sums fit one word (allele bits from bit
        // 22, sum v from bit 11, sum w), one add per allele; below 2^16: 32-bit sums (a row's
        // 256 items stay below 2^24); else 64-bit ones. Uniform over the warp.
        const int form = __all_sync(0xffffffffu, any < 0x100u) ? 0 : __all_sync(0xffffffffu, any < 0x10000u) ? 1 : 2;
        if (form == 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) w[i] |= (v[i] << 11) | (1 << (22 + i));
        }
        auto load_row = [&](int32_t c) -> uint4 {
            const size_t row = (size_t)c * a.ng;
            if (nv == 8) return load_half8(a.k, row + j0, total);
            uint32_t q[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int i = 0; i < 7; ++i)
                if (i < nv) q[i >> 1] |= (uint32_t)(uint16_t)a.k[row + j0 + i] << (16 * (i & 1));
            return make_uint4(q[0], q[1], q[2], q[3]);
        };
        uint4 hn = load_row((int32_t)c_begin);
        for (int32_t c = (int32_t)c_begin; c < c_end; ++c) {
            const size_t row = (size_t)c * a.ng;
            const uint4 h = hn;
            if (c + 1 < c_end) hn = load_row(c + 1);        // in flight while this row is computed
            // angle indices outside [-K, K] are invalid input; they are clamped so that the
            // table lookup stays inside the table; 4(k + K) is T's byte offset
            uint32_t sp[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) sp[i] = __vadd2(__vmins2(__vmaxs2(sp[i], kneg), kk), kk) << 2;
            const qieo::Draw4 d0 = qieo::philox4x32_10((uint32_t)(j0 / 4u), (uint32_t)c, (uint32_t)a.t, 0u, a.seed, a.inst);
            const qieo::Draw4 d1 = qieo::philox4x32_10((uint32_t)(j0 / 4u) + 1u, (uint32_t)c, (uint32_t)a.t, 0u, a.seed, a.inst);
            const uint32_t u[8] = {d0.a, d0.b, d0.c, d0.d, d1.a, d1.b, d1.c, d1.d};
            uint32_t xbits;
            long long sw, sv;
            bool x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t off = (i & 1) ? (sp[i >> 1] >> 16) : (sp[i >> 1] & 0xffffu);
                x[i] = u[i] < *reinterpret_cast<const uint32_t *>(thr_bytes + off) || off == off_top;
            }
            // the sums (items past the row's end are 0)
            if (form == 0) {
                uint32_t acc = 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (x[i]) acc += (uint32_t)w[i];
                xbits = acc >> 22;
                const uint32_t both = __reduce_add_sync(0xffffffffu, (acc & 0x7ffu) | ((acc & 0x3ff800u) << 5));
                sw = (long long)(both & 0xffffu);
                sv = (long long)(both >> 16);
            } else {
                xbits = 0u;
                if (form == 1) {
                    uint32_t lw = 0u, lv = 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (x[i]) {
                            xbits |= 1u << i;
                            lw += (uint32_t)w[i];
                            lv += (uint32_t)v[i];
                        }
                    sw = (long long)__reduce_add_sync(0xffffffffu, lw);
                    sv = (long long)__reduce_add_sync(0xffffffffu, lv);
                } else {
                    long long lw = 0, lv = 0;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (x[i]) {
                            xbits |= 1u << i;
                            lw += w[i];
                            lv += v[i];
                        }
                    sw = warp_sum(lw);
                    sv = warp_sum(lv);
                }
            }
            if (lane < 2)
                atomicAdd(reinterpret_cast<unsigned long long *>(a.sums + 2 * (size_t)c + lane),
                          (unsigned long long)(lane ? sv : sw));
            // the alleles as bytes: the multiplier moves bit i of a nibble to bit 8i, and the
            // sixteen partial products all land on different bits
            const uint32_t b0 = ((xbits & 15u) * 0x00204081u) & 0x01010101u;
            const uint32_t b1 = ((xbits >> 4) * 0x00204081u) & 0x01010101u;
            // the alleles: lane l stores the aligned word that starts b bytes before its own
            uint8_t *const xp = a.x + row + j0;
            const uint32_t b = (uint32_t)(reinterpret_cast<uintptr_t>(xp) & 7u);
            if (b == 0u) {
                if (nv == 8) {
                    *reinterpret_cast<uint2 *>(xp) = make_uint2(b0, b1);
                } else {
#pragma unroll
                    for (int i = 0; i < 7; ++i)
                        if (i < nv) xp[i] = (uint8_t)((i < 4 ? b0 : b1) >> (8 * (i & 3)));
                }
            } else {
                const uint64_t own = (uint64_t)b0 | ((uint64_t)b1 << 32);
                const uint64_t prev = __shfl_up_sync(0xffffffffu, own, 1);
                const bool last = lane == 31 || left <= 8;   // no lane after this one holds genes
                if (lane > 0 && nv == 8)
                    *reinterpret_cast<uint64_t *>(xp - b) = (prev >> (64u - 8u * b)) | (own << (8u * b));
                if (lane == 0 && nv == 8) {                 // up to the next aligned word
                    const uint32_t n = 8u - b;
                    uint64_t v8 = own;
                    uint8_t *q = xp;
                    if (n & 1u) {
                        *q = (uint8_t)v8;
                        q += 1;
                        v8 >>= 8;
                    }
                    if (n & 2u) {
                        *reinterpret_cast<uint16_t *>(q) = (uint16_t)v8;
                        q += 2;
                        v8 >>= 16;
                    }
                    if (n & 4u) *reinterpret_cast<uint32_t *>(q) = (uint32_t)v8;
                }
                if (nv == 8 && last) {                      // the last b bytes, with no lane after
                    uint64_t v8 = own >> (64u - 8u * b);
                    uint8_t *q = xp + (8u - b);
                    if (b & 4u) {
                        *reinterpret_cast<uint32_t *>(q) = (uint32_t)v8;
                        q += 4;
                        v8 >>= 32;
                    }
                    if (b & 2u) {
                        *reinterpret_cast<uint16_t *>(q) = (uint16_t)v8;
                        q += 2;
                        v8 >>= 16;
                    }
                    if (b & 1u) *q = (uint8_t)v8;
                }
                if (nv > 0 && nv < 8) {                     // the row's last genes
                    if (lane > 0)                           // the previous lane's last b bytes
                        for (uint32_t i = 0; i < b; ++i)
                            xp[(int)i - (int)b] = (uint8_t)(prev >> (64u - 8u * b + 8u * i));
                    for (int i = 0; i < nv; ++i) xp[i] = (uint8_t)(own >> (8 * i));
                }
            }
        }
    }

    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == gridDim.x - 1u;
    allow_dependent_launch();
    __syncthreads();
    if (!s_last) return;
    __threadfence();

    int64_t bf = INT64_MIN;
    int32_t bc = 0x7fffffff;
    auto take = [&](int c, longlong2 s) {
        const int64_t f = s.x <= a.capacity ? s.y : -a.lambda * (s.x - a.capacity);
        a.fitness[c] = f;
        if (f > bf) {
            bf = f;
            bc = c;
        }
    };
    const longlong2 *sums = reinterpret_cast<const longlong2 *>(a.sums);
    int c = threadIdx.x;
    for (; c + 7 * kThreads < a.np; c += 8 * kThreads) {    // eight loads in flight
        longlong2 s[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) s[i] = __ldcg(sums + c + i * kThreads);
#pragma unroll
        for (int i = 0; i < 8; ++i) take(c + i * kThreads, s[i]);
    }
    for (; c < a.np; c += kThreads) take(c, __ldcg(sums + c));
    for (int o = 16; o > 0; o >>= 1) {
        const int64_t of = __shfl_xor_sync(0xffffffffu, bf, o);
        const int32_t oc = __shfl_xor_sync(0xffffffffu, bc, o);
        if (of > bf || (of == bf && oc < bc)) {
            bf = of;
            bc = oc;
        }
    }
    if ((threadIdx.x & 31) == 0) {
        s_f[threadIdx.x >> 5] = bf;
        s_c[threadIdx.x >> 5] = bc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kThreads / 32; ++w)
            if (s_f[w] > bf || (s_f[w] == bf && s_c[w] < bc)) {
                bf = s_f[w];
                bc = s_c[w];
            }
        *a.elite = bc;
    }
}

// CIP of generation t: every angle index one step toward the elite's allele (rule R1), or
// only where the allele differs from the elite's (rule R2), saturating at -K and K. The
// buffer is walked in aligned 16-byte chunks whatever the rows' alignment, each with the
// elite's 8 alleles of its columns; the elements before the first and after the last whole
// chunk, and chunks that span two rows, go one by one. Bound by memory (4 B a gene under R1,
// 5 under R2).
template <int kRule>
__device__ __forceinline__ void noalloc_step(int16_t *k, const uint8_t *x, const uint8_t *xe, int32_t K,
                                             size_t idx, uint32_t j)
{
    const int xe_j = xe[j];
    if (kRule == 1 && x[idx] == xe_j) return;
    const int32_t kn = (int32_t)k[idx] + (xe_j ? 1 : -1);
    if (kn >= -K && kn <= K) k[idx] = (int16_t)kn;
}

template <int kRule>
__global__ void __launch_bounds__(kThreads) noalloc_cip_kernel(int16_t *k, const uint8_t *x, const int32_t *elite,
                                                               int32_t np, int32_t ng, int32_t K)
{
    grid_dependency_wait();
    const size_t total = (size_t)np * ng;
    const size_t head = min(total, (size_t)(((16u - (uint32_t)(reinterpret_cast<uintptr_t>(k) & 15u)) & 15u) / 2u));
    const size_t chunks = (total - head) / 8;
    const size_t tid = (size_t)blockIdx.x * kThreads + threadIdx.x, stride = (size_t)gridDim.x * kThreads;
    const size_t xe0 = (size_t)*elite * ng;
    const uint8_t *xe = x + xe0;
    // column of this thread's chunk, advanced by the stride without divisions
    size_t f = head + 8 * tid;
    uint32_t j = (uint32_t)(f % (size_t)ng);
    const uint32_t jstep = (uint32_t)(8 * stride % (size_t)ng);
    const uint32_t kk = (uint32_t)K * 0x00010001u, kneg = __vneg2(kk);
    for (size_t i = tid; i < chunks; i += stride) {
        if (j + 8u <= (uint32_t)ng) {
            const uint4 h = *reinterpret_cast<const uint4 *>(k + f);
            const uint2 e = load_byte8(x, xe0 + j, total);
            const uint2 o = kRule == 1 ? load_byte8(x, f, total) : make_uint2(0u, 0u);
            const uint32_t kp[4] = {h.x, h.y, h.z, h.w};
            uint32_t r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t e2 = __byte_perm(q < 2 ? e.x : e.y, 0u, (q & 1) ? 0x4342 : 0x4140);
                uint32_t step = __vsub2(e2 << 1, 0x00010001u);            // +1 or -1 per half
                if (kRule == 1) {
                    const uint32_t o2 = __byte_perm(q < 2 ? o.x : o.y, 0u, (q & 1) ? 0x4342 : 0x4140);
                    step &= (e2 ^ o2) * 0xffffu;                          // 0 where the alleles agree
                }
                const uint32_t kn = __vadd2(kp[q], step);
                const uint32_t in = __vcmpeq2(__vmins2(__vmaxs2(kn, kneg), kk), kn);
                r[q] = (kn & in) | (kp[q] & ~in);
            }
            *reinterpret_cast<uint4 *>(k + f) = make_uint4(r[0], r[1], r[2], r[3]);
        } else {
            uint32_t jj = j;
            for (int q = 0; q < 8; ++q) {
                noalloc_step<kRule>(k, x, xe, K, f + q, jj);
                if (++jj == (uint32_t)ng) jj = 0u;
            }
        }
        f += 8 * stride;
        j += jstep;
        if (j >= (uint32_t)ng) j -= (uint32_t)ng;
    }
    // elements before the first and after the last chunk
    const size_t tail0 = head + 8 * chunks, loose = head + (total - tail0);
    if (tid < loose) {
        const size_t idx = tid < head ? tid : tail0 + (tid - head);
        noalloc_step<kRule>(k, x, xe, K, idx, (uint32_t)(idx % (size_t)ng));
    }
}

// Device address of g_noalloc_scratch on the current device (looked up once per device).
qieo_status scratch_address(unsigned char **out, int *device)
{
    int dev = 0;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess) return noalloc_fail(QIEO_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(ce));
    if (dev < 0 || dev >= kMaxDevices) return noalloc_fail(QIEO_ERR_INVALID, "device %d out of range", dev);
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr;
        ce = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (ce != cudaSuccess || !p)
            return noalloc_fail(QIEO_ERR_CUDA, "cudaGetSymbolAddress(g_noalloc_scratch): %s",
                                cudaGetErrorString(ce));
        g_scratch_ptr[dev] = static_cast<unsigned char *>(p);
    }
    *out = g_scratch_ptr[dev];
    *device = dev;
    return QIEO_OK;
}

// T[n] = round(sin^2(n pi / D) 2^32) = round(2^31 (1 - cos(2 pi n / D))) for n <= K,
// mirrored above (T[2K - n] = 2^32 - T[n]); T[0] = 0 and T[K] = 2^31 exactly. The last
// few tables are kept per step count (26 extended-precision cosines cost more than the
// launches of a small call).
void fill_thresholds(int32_t D, uint32_t *thr)
{
    struct Table {
        int32_t D = 0;
        uint32_t thr[kMaxThr];
    };
    constexpr int kTables = 4;
    static std::mutex mu;
    static Table tables[kTables];
    static int next = 0;
    const int32_t K = D / 4;
    std::lock_guard<std::mutex> lock(mu);
    for (const Table &t : tables)
        if (t.D == D) {
            std::memcpy(thr, t.thr, (size_t)(2 * K + 1) * sizeof(uint32_t));
            return;
        }
    Table &t = tables[next];
    next = (next + 1) % kTables;
    t.D = 0;
    const long double pi = acosl(-1.0L);
    for (int32_t n = 0; n <= K; ++n) {
        const long double val = 2147483648.0L * (1.0L - cosl(2.0L * pi * n / D));
        t.thr[n] = (uint32_t)llroundl(val);
    }
    t.thr[0] = 0u;
    t.thr[K] = 1u << 31;
    for (int32_t n = K + 1; n <= 2 * K; ++n) t.thr[n] = (uint32_t)((1ull << 32) - t.thr[2 * K - n]);
    t.D = D;
    std::memcpy(thr, t.thr, (size_t)(2 * K + 1) * sizeof(uint32_t));
}

// The three launches of a call: the sums cleared, observation with the elite, rotation.
// Each may start while the one before drains (programmatic dependent launch).
template <int kThr>
qieo_status launch_noalloc(const qieo_problem &problem, const qieo_params &params, int32_t t, int16_t *k, uint8_t *x,
                           int64_t *fitness, int32_t *elite, unsigned char *scratch, int sms)
{
    const int32_t ng = problem.ng, np = params.np;
    NoallocArgs<kThr> a;
    std::memset(&a, 0, sizeof a);
    a.w = problem.weights;
    a.v = problem.values;
    a.k = k;
    a.x = x;
    a.fitness = fitness;
    a.elite = elite;
    a.counter = reinterpret_cast<unsigned int *>(scratch);
    a.sums = reinterpret_cast<long long *>(scratch + kCounterBytes);
    a.capacity = problem.capacity;
    a.lambda = params.penalty_lambda;
    a.ng = ng;
    a.np = np;
    a.K = params.dtheta_den / 4;
    a.t = t;
    a.seed = params.seed;
    a.inst = params.instance_id;
    fill_thresholds(params.dtheta_den, a.thr);
    // Rows per warp: one wave of the 24 warps an SM holds, and at most 64 rows (the items are
    // then loaded once per 16,384 genes).
    a.ntile = (int32_t)(((int64_t)ng + kTileGenes - 1) / kTileGenes);
    const int64_t units = (int64_t)a.ntile * np, warps = (int64_t)24 * sms;
    a.rows = (int32_t)std::max<int64_t>(1, std::min<int64_t>(64, (units + warps - 1) / warps));
    const int64_t items = (int64_t)a.ntile * (((int64_t)np + a.rows - 1) / a.rows);
    const int64_t obs_blocks = (items + kThreads / 32 - 1) / (kThreads / 32);

    cudaStream_t s = static_cast<cudaStream_t>(params.stream);
    const int clear_blocks = (int)std::min<int64_t>(((int64_t)2 * np + kThreads - 1) / kThreads, 1024);
    noalloc_clear_kernel<<<clear_blocks, kThreads, 0, s>>>(a.counter, a.sums, 2 * np);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)obs_blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t ce = cudaGetLastError();
    if (ce == cudaSuccess) ce = cudaLaunchKernelEx(&cfg, noalloc_observe_kernel<kThr>, a);
    const int64_t chunks = (int64_t)np * ng / 8 + 16;
    cfg.gridDim = dim3((unsigned int)std::max<int64_t>(1, std::min<int64_t>((chunks + kThreads - 1) / kThreads, 8 * (int64_t)sms)));
    if (ce == cudaSuccess)
        ce = params.rotate_rule == 1
                 ? cudaLaunchKernelEx(&cfg, noalloc_cip_kernel<1>, k, (const uint8_t *)x, (const int32_t *)elite, np, ng, a.K)
                 : cudaLaunchKernelEx(&cfg, noalloc_cip_kernel<0>, k, (const uint8_t *)x, (const int32_t *)elite, np, ng, a.K);
    if (ce != cudaSuccess) return noalloc_fail(QIEO_ERR_CUDA, "launch: %s", cudaGetErrorString(ce));
    return QIEO_OK;
}

}  // namespace

namespace qieo_internal {
// The threshold words for the library's other translation units ([2 (D / 4) + 1]).
void fill_thresholds(int32_t D, uint32_t *thr) { ::fill_thresholds(D, thr); }
}  // namespace qieo_internal

extern "C" qieo_status qieo_generation_noalloc(const qieo_problem *problem, const qieo_params *params,
                                               int32_t t, int16_t *k, uint8_t *x, int64_t *fitness,
                                               int32_t *elite)
{
    if (!problem || !params || !k || !x || !fitness || !elite || !problem->weights || !problem->values)
        return noalloc_fail(QIEO_ERR_INVALID, "NULL argument");
    const int32_t ng = problem->ng, np = params->np, D = params->dtheta_den;
    if (ng < 1) return noalloc_fail(QIEO_ERR_INVALID, "ng must be >= 1 (got %d)", ng);
    if (np < 1 || np > QIEO_NOALLOC_MAX_NP)
        return noalloc_fail(QIEO_ERR_INVALID,
                            "np must be in [1, %d] (the size of the static scratch array); got %d",
                            QIEO_NOALLOC_MAX_NP, np);
    if (D < 4 || D > kMaxD || D % 4 != 0)
        return noalloc_fail(QIEO_ERR_INVALID, "dtheta_den must be a multiple of 4 in [4, %d]", kMaxD);
    if (params->penalty_lambda < 1) return noalloc_fail(QIEO_ERR_INVALID, "penalty_lambda must be >= 1");
    if (params->rotate_rule != QIEO_RULE_R1 && params->rotate_rule != QIEO_RULE_R2)
        return noalloc_fail(QIEO_ERR_INVALID, "rotate_rule must be 0 or 1");
    if (problem->capacity < 0) return noalloc_fail(QIEO_ERR_INVALID, "capacity must be >= 0");
    if (t < 0) return noalloc_fail(QIEO_ERR_INVALID, "generation t must be >= 0");
    if ((int64_t)np * ng > ((int64_t)1 << 40)) return noalloc_fail(QIEO_ERR_INVALID, "np * ng too large");

    unsigned char *scratch = nullptr;
    int dev = 0;
    qieo_status st = scratch_address(&scratch, &dev);
    if (st != QIEO_OK) return st;

    int sms = 0;
    cudaError_t ce = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (ce != cudaSuccess) return noalloc_fail(QIEO_ERR_CUDA, "device query: %s", cudaGetErrorString(ce));
    return D / 2 + 1 <= kSmallThr ? launch_noalloc<kSmallThr>(*problem, *params, t, k, x, fitness, elite, scratch, sms)
                                  : launch_noalloc<kMaxThr>(*problem, *params, t, k, x, fitness, elite, scratch, sms);
}
