// vcm_kernels.cu -- sm_103a kernels of the visibility color map engine.
//
//  * grid build: boxes bucketed by footprint centre into a uniform 2D grid
//    (count -> scan -> scatter -> permuted copies in box order -> bounds);
//  * tile pass: persistent blocks draw viewpoint tiles from a queue; each tile
//    culls the scene against the convex hull of (tile, target) using the
//    grid, stages the candidates in shared memory with cp.async, decides the
//    viewpoints that one box hides, and publishes the others;
//  * sweep: warps take the published viewpoints, lanes over target patch columns
//    and bits of a mask over patch rows, deciding each viewpoint->patch segment
//    by float32 slab intervals (Def. 2 point-to-point visibility; touching
//    blocks, Def. 4) with an exact integer re-decision inside a 1e-6 margin
//    band, then summing A cos(theta)/d^2 (or len cos(theta)/d in 2D);
//  * quantise: colors in L levels from v / v_ref (Def. 1 normalisation).
#include "vcm_internal.h"

#include <cfloat>
#include <climits>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <utility>

namespace vcm {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// The kernels of a call follow one another closely, so each is launched ahead of
// the end of the one before it (programmatic stream serialization) and waits
// here until that one has completed with its writes visible.  Every thread of
// every kernel waits, so a kernel's end implies those before it.  The kernel
// before lets go when its blocks exit: letting go at its start put waiting
// blocks beside the persistent passes (64 uneven requests +1 %).  Without the
// launch attribute this does nothing.  512^2 x 5 viewpoints, 5,000 boxes: 126 ->
// 117 us per call; a 2D map of 128 x 128 36 -> 28 us.
__device__ __forceinline__ void after_previous_kernel()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ float f_inf() { return __int_as_float(0x7f800000); }

// Bounds checks of the checked build (libvcm_checked, compiled with
// VCM_CHECKED): an index outside its buffer sets the request's error word to
// VCM_DEVERR_BOUNDS and the access is skipped; nothing traps.  In the normal
// build the check is the constant true and costs nothing.
#ifdef VCM_CHECKED
__device__ __noinline__ bool in_bounds_slow(long long i, long long n, vcm_stats *st)
{
    if (i >= 0 && i < n)
        return true;
    if (st)
        atomicExch(&st->error, (unsigned)VCM_DEVERR_BOUNDS);
    return false;
}
#define IN_BOUNDS(i, n, st) in_bounds_slow((long long)(i), (long long)(n), (st))
#define CHECKED(ok, st) in_bounds_slow((ok) ? 0 : 1, 1, (st))   // the same for a rule of vcm_internal.h
#else
#define IN_BOUNDS(i, n, st) true
#define CHECKED(ok, st) true
#endif

// The ids of a candidate list past its staged boxes: ints, or 3 bytes each in a
// spill region (scenes of less than 2^24 boxes: 8 blocks per SM then spill
// into what 6 blocks needed with ints).
struct Tail {
    const void *p;
    int bytes;
    __device__ __forceinline__ int operator[](int i) const
    {
        if (bytes == 4)
            return static_cast<const int *>(p)[i];
        const unsigned char *b = static_cast<const unsigned char *>(p) + 3 * (size_t)i;
        return (int)(b[0] | (b[1] << 8) | (b[2] << 16));
    }
    __device__ __forceinline__ void put(int i, int id) const
    {
        if (bytes == 4) {
            static_cast<int *>(const_cast<void *>(p))[i] = id;
            return;
        }
        unsigned char *b = static_cast<unsigned char *>(const_cast<void *>(p)) + 3 * (size_t)i;
        b[0] = (unsigned char)id;
        b[1] = (unsigned char)(id >> 8);
        b[2] = (unsigned char)(id >> 16);
    }
};

// Box i of a tile's candidate list: staged in shared memory, or (past
// n_smem) through its id in the list's tail.  The checked build
// replaces an out-of-range id by an empty box, which blocks nothing.
__device__ __forceinline__ void load_box(const float4 *__restrict__ sbox, int n_smem, Tail spill,
                                         const float4 *__restrict__ gbox, int i, int n_boxes, vcm_stats *st,
                                         float4 &lo, float4 &hi)
{
    if (i < n_smem) {
        lo = sbox[2 * i];
        hi = sbox[2 * i + 1];
        return;
    }
    const int s = IN_BOUNDS(i - n_smem, n_boxes, st) ? spill[i - n_smem] : -1;
    if (!IN_BOUNDS(s, n_boxes, st)) {
        lo = make_float4(f_inf(), f_inf(), f_inf(), 0.f);
        hi = make_float4(-f_inf(), -f_inf(), -f_inf(), 0.f);
        return;
    }
    lo = __ldg(&gbox[2 * s]);
    hi = __ldg(&gbox[2 * s + 1]);
}

// Output stores of a request: value of viewpoint vp, occlusion-bit word at
// index `at` (bounds checked in the checked build).
__device__ __forceinline__ void put_v(const DevRequest &R, long long vp, float v)
{
    if (IN_BOUNDS(vp, (long long)R.nx * R.ny * R.nl, R.stats))
        R.v_out[vp] = v;
}
__device__ __forceinline__ void put_word(const DevRequest &R, long long at, uint32_t w)
{
    if (IN_BOUNDS(at, (long long)R.nx * R.ny * R.nl * R.words, R.stats))
        R.bits_out[at] = w;
}

// Hardware reciprocal, at most 1 ulp from 1/d (2^-23 relative); 1/(+0) = +inf.
// The slab-test error bound with it is about 5 u per t value, 10 u per
// margin, still inside the 1e-6 band that is re-decided exactly.
__device__ __forceinline__ float rcp_approx(float d)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return r;
}

// rsqrtf without its scaling of subnormal arguments: squared distances of
// distinct lattice points are at least 2^-20 m^2.
__device__ __forceinline__ float rsqrt_normal(float d2)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d2));
    return r;
}

// Two floats per operation (each rounded as the scalar one).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 x, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// ---------------------------------------------------------------------------
// grid build
// ---------------------------------------------------------------------------

__global__ void k_box_cell(const float *__restrict__ lo, const float *__restrict__ hi, int n,
                           float gx0, float gy0, float inv_cell, int gnx, int gny,
                           int *__restrict__ cell_of, int *__restrict__ count)
{
    after_previous_kernel();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    float cx = 0.5f * (lo[3 * i + 0] + hi[3 * i + 0]);
    float cy = 0.5f * (lo[3 * i + 1] + hi[3 * i + 1]);
    int ix = (int)floorf((cx - gx0) * inv_cell);
    int iy = (int)floorf((cy - gy0) * inv_cell);
    ix = min(max(ix, 0), gnx - 1);
    iy = min(max(iy, 0), gny - 1);
    int c = iy * gnx + ix;
    cell_of[i] = c;
    atomicAdd(&count[c], 1);
}

// Exclusive scan of count[0..n) into start[0..n] by one block, for at most
// kScanOneMax cells: 4,096 a round, 4 per thread.  At these sizes the three
// kernels below are three launch latencies (15 us against 5).
constexpr int kScanOneThreads = 1024;
constexpr int kScanOneMax = 65536;
__global__ void __launch_bounds__(kScanOneThreads) k_scan_one(const int *__restrict__ count, int n,
                                                              int *__restrict__ start,
                                                              unsigned *__restrict__ overhang_bits)
{
    after_previous_kernel();
    __shared__ int s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int carry = 0;
    for (int base = 0; base < n; base += 4 * kScanOneThreads) {
        const int i = base + 4 * threadIdx.x;
        int v[4], local = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = i + k < n ? count[i + k] : 0;
            local += v[k];
        }
        int incl = local;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int t = __shfl_up_sync(kFull, incl, off);
            if (lane >= off)
                incl += t;
        }
        if (lane == 31)
            s_warp[warp] = incl;
        __syncthreads();
        const int w = s_warp[lane];
        int wincl = w;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int t = __shfl_up_sync(kFull, wincl, off);
            if (lane >= off)
                wincl += t;
        }
        int run = carry + incl - local + __shfl_sync(kFull, wincl - w, warp);
        carry += __shfl_sync(kFull, wincl, 31);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < n)
                start[i + k] = run;
            run += v[k];
        }
        __syncthreads();   // s_warp is reused
    }
    if (threadIdx.x == 0) {
        start[n] = carry;
        *overhang_bits = 0u;   // k_cell_bounds accumulates it
    }
}

// Exclusive scan of count[0..n) into start[0..n] in three kernels: block
// sums of kScanChunk elements, a one-block scan of the block sums (at most
// 1024 of them: n <= 4M cells), then each block's scan with its offset.
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanChunk = kScanThreads * kScanItems;   // 4096 elements per block

// Exclusive scan of one int per thread over a block of kScanThreads;
// returns the thread's prefix and sets total.
__device__ __forceinline__ int block_exclusive_scan(int x, int &total)
{
    __shared__ int s_warp[kScanThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, off);
        if (lane >= off)
            incl += t;
    }
    if (lane == 31)
        s_warp[warp] = incl;
    __syncthreads();
    int before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) {
        before += w < warp ? s_warp[w] : 0;
        total += s_warp[w];
    }
    __syncthreads();   // s_warp may be reused by the caller's next scan
    return before + incl - x;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const int *__restrict__ count, int n,
                                                              int *__restrict__ block_sum)
{
    after_previous_kernel();
    const int base = blockIdx.x * kScanChunk;
    int local = 0;
    for (int i = threadIdx.x; i < kScanChunk && base + i < n; i += kScanThreads)
        local += count[base + i];
    int total;
    (void)block_exclusive_scan(local, total);
    if (threadIdx.x == 0)
        block_sum[blockIdx.x] = total;
}

// One block: exclusive scan of the n_blocks (<= 1024) block sums in place;
// start[n] gets the grand total.
__global__ void __launch_bounds__(1024) k_scan_top(int *__restrict__ block_sum, int n_blocks, int n,
                                                   int *__restrict__ start, unsigned *__restrict__ overhang_bits)
{
    after_previous_kernel();
    __shared__ int s_part[1024];
    const int t = threadIdx.x;
    const int x = t < n_blocks ? block_sum[t] : 0;
    s_part[t] = x;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const int v = t >= off ? s_part[t - off] : 0;
        __syncthreads();
        s_part[t] += v;
        __syncthreads();
    }
    if (t < n_blocks)
        block_sum[t] = s_part[t] - x;
    if (t == 1023) {
        start[n] = s_part[t];
        *overhang_bits = 0u;   // k_cell_bounds accumulates it
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_down(const int *__restrict__ count, int n,
                                                            const int *__restrict__ block_off, int *__restrict__ start)
{
    after_previous_kernel();
    // each thread owns kScanItems consecutive elements of the block's chunk
    const int base = blockIdx.x * kScanChunk + threadIdx.x * kScanItems;
    int v[kScanItems], local = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < n ? count[base + k] : 0;
        local += v[k];
    }
    int total;
    int run = block_off[blockIdx.x] + block_exclusive_scan(local, total);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n)
            start[base + k] = run;
        run += v[k];
    }
}

// Each box takes a place in its cell, in any order (the counts run down to 0).
__global__ void k_scatter(const int *__restrict__ cell_of, int n, const int *__restrict__ start,
                          int *__restrict__ count, int *__restrict__ order)
{
    after_previous_kernel();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    int c = cell_of[i];
    order[start[c] + atomicSub(&count[c], 1) - 1] = i;
}

struct PermPtrs {
    float4 *p[6];
};

// The permuted copies, in ascending box index inside each cell (the scatter's
// atomics leave the order arbitrary): a box's place is the number of smaller
// indices in its cell, counted by its thread.  Cells hold a few boxes, and in a
// crowded one the threads of a warp read the same list.  (Sorting the cells in
// place first, a thread each, was a kernel of 18 us of dependent loads.)
__global__ void k_write_boxes(const float *__restrict__ lo, const float *__restrict__ hi, int n,
                              const int *__restrict__ cell_of, const int *__restrict__ start,
                              const int *__restrict__ order, PermPtrs out)
{
    after_previous_kernel();
    int at = blockIdx.x * blockDim.x + threadIdx.x;
    if (at >= n)
        return;
    const int id = order[at], c = cell_of[id];
    const int b = start[c], e = start[c + 1];
    const float L[3] = {lo[3 * id], lo[3 * id + 1], lo[3 * id + 2]};
    const float H[3] = {hi[3 * id], hi[3 * id + 1], hi[3 * id + 2]};
    int s = b;
    for (int j = b; j < e; ++j)
        s += order[j] < id;
#pragma unroll
    for (int p = 0; p < 6; ++p) {
        const int a0 = p >> 1, a1 = (p & 1) ? (a0 == 2 ? 1 : 2) : (a0 == 0 ? 1 : 0), a2 = 3 - a0 - a1;
        out.p[p][2 * s] = make_float4(L[a0], L[a1], L[a2], __int_as_float(id));
        out.p[p][2 * s + 1] = make_float4(H[a0], H[a1], H[a2], 0.f);
    }
}

__global__ void k_cell_bounds(const float4 *__restrict__ boxes, const int *__restrict__ start,
                              int gnx, int gny, float gx0, float gy0, float cell,
                              float4 *__restrict__ cell_lo, float4 *__restrict__ cell_hi,
                              unsigned *__restrict__ overhang_bits)
{
    after_previous_kernel();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = c < gnx * gny;
    float4 lo = make_float4(f_inf(), f_inf(), f_inf(), 0.f);
    float4 hi = make_float4(-f_inf(), -f_inf(), -f_inf(), 0.f);
    const int b = in ? start[c] : 0, e = in ? start[c + 1] : 0;
    for (int s = b; s < e; ++s) {
        float4 l = boxes[2 * s], h = boxes[2 * s + 1];
        lo.x = fminf(lo.x, l.x); lo.y = fminf(lo.y, l.y); lo.z = fminf(lo.z, l.z);
        hi.x = fmaxf(hi.x, h.x); hi.y = fmaxf(hi.y, h.y); hi.z = fmaxf(hi.z, h.z);
    }
    if (in) {
        cell_lo[c] = lo;
        cell_hi[c] = hi;
    }
    float oh = 0.f;
    if (e > b) {
        const int ix = c % gnx, iy = c / gnx;
        const float x0 = gx0 + ix * cell, y0 = gy0 + iy * cell;
        oh = fmaxf(fmaxf(x0 - lo.x, hi.x - (x0 + cell)), fmaxf(y0 - lo.y, hi.y - (y0 + cell)));
        oh = fmaxf(oh, 0.f);
    }
    const unsigned most = __reduce_max_sync(kFull, __float_as_uint(oh));
    if ((threadIdx.x & 31) == 0 && most)
        atomicMax(overhang_bits, most);
}

// ---------------------------------------------------------------------------
// tile kernel
// ---------------------------------------------------------------------------

__device__ __forceinline__ float4 world_box_lo(const DevScene &sc, int s) { return __ldg(&sc.boxes[0][2 * s]); }
__device__ __forceinline__ float4 world_box_hi(const DevScene &sc, int s) { return __ldg(&sc.boxes[0][2 * s + 1]); }

// The union of every segment from a tile's viewpoints A to the target's patch
// rectangle B, both axis-aligned boxes: conv(A, B), which is the union over t
// in [0, 1] of the boxes (1 - t) A + t B.  An axis-aligned box [lo, hi] meets it
// iff some t in [0, 1] satisfies, on each axis,
//     t (B_hi - A_hi) >= lo - A_hi   and   t (B_lo - A_lo) <= hi - A_lo,
// six linear bounds on t.  Each is an entry (t >= m e + o) or an exit (t <= m e
// + o) of the box's edge e by the sign of its slope; the other one gets m = 0
// and an infinite o, so a test is 12 fused multiply-adds and as many minima,
// without a branch.  A and B are widened by 0.04 m, more than ten times the
// rounding of an edge's bound in metres at 16,384 m (about 2^-24 x 16384 x 3),
// so a box that meets the hull is never dropped.
//
// The separating planes of the hull that this replaces took 56 candidate normals
// per tile and up to 20 plane tests per box, and dropped fewer boxes.  Tile
// kernels before and after: 512^2 x 5 viewpoints, 5,000 boxes 0.164 -> 0.150 ms
// (viewer-centric 0.107 -> 0.079 ms); 2,048^2 x 8, 100,000 boxes 5.20 -> 4.63 ms
// (the tile pass 2.47 -> 1.91 ms); 64 uneven requests 8.72 -> 8.30 ms.
struct Swept {
    float m[6][2], o[6][2];   // bound (axis, lo or hi edge): entry, exit
};
// Slopes below this many metres count as 0: the bound then holds for every t
// or for none.
__device__ __forceinline__ void swept_bound(Swept &S, int k, float a, float b, bool upper_edge)
{
    const float d = b - a;
    const float inv = fabsf(d) < 1e-3f ? 1e30f : rcp_approx(d);
    const bool entry = (fabsf(d) < 1e-3f || d > 0.f) != upper_edge;
    S.m[k][0] = entry ? inv : 0.f;
    S.o[k][0] = entry ? -a * inv : -f_inf();
    S.m[k][1] = entry ? 0.f : inv;
    S.o[k][1] = entry ? f_inf() : -a * inv;
}
__device__ __forceinline__ Swept make_swept(const float (*A)[2], const float (*B)[2])
{
    constexpr float kPad = 0.04f;
    Swept S;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        swept_bound(S, 2 * ax, A[ax][1] + kPad, B[ax][1] + kPad, false);   // lower edge against the upper sides
        swept_bound(S, 2 * ax + 1, A[ax][0] - kPad, B[ax][0] - kPad, true);
    }
    return S;
}
__device__ __forceinline__ bool swept_meets(const Swept &S, float4 lo, float4 hi)
{
    const float e[6] = {lo.x, hi.x, lo.y, hi.y, lo.z, hi.z};
    float from = 0.f, to = 1.f;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        from = fmaxf(from, fmaf(e[k], S.m[k][0], S.o[k][0]));
        to = fminf(to, fmaf(e[k], S.m[k][1], S.o[k][1]));
    }
    return from <= to;
}

// Exact re-decision of one segment against one box, in integers.  Inputs are
// lattice values (multiples of 2^-10 m, |x| <= 2^14 m): in lattice units their
// differences take 26 bits and a product of two of them 52, so the comparisons
// below are exact.  The running lower bound en/ed and upper bound xn/xd of the
// segment parameter t are kept as fractions with positive denominators.  (The
// same in float64 is exact too, but took 2.8 us per call on the narrow FP64
// pipe, and a column that grazes a box asked for 16 to 32 of them in a row:
// 1 % of the sweep's warps set its end.  512^2 x 5 viewpoints, 5,000 boxes: both
// passes 128 -> 105 us, strict 101 -> 68 us.)
__device__ __noinline__ bool exact_hit(float qu, float qn, float qw, float pu, float pn, float pw,
                                       float4 lo, float4 hi)
{
    constexpr float kUnits = (float)VCM_UNITS_PER_M;
    const float q[3] = {qu, qn, qw};
    const float p[3] = {pu, pn, pw};
    const float L[3] = {lo.x, lo.y, lo.z};
    const float H[3] = {hi.x, hi.y, hi.z};
    int en = 0, ed = 1, xn = 1, xd = 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int at = __float2int_rn(q[k] * kUnits);
        const int d = __float2int_rn(p[k] * kUnits) - at;
        const int a = __float2int_rn(L[k] * kUnits) - at;
        const int b = __float2int_rn(H[k] * kUnits) - at;
        if (d == 0) {
            if (a > 0 || b < 0)
                return false;
            continue;
        }
        const int ln = d > 0 ? a : -b, un = d > 0 ? b : -a, den = abs(d);
        if ((long long)ln * ed > (long long)en * den) {
            en = ln;
            ed = den;
        }
        if ((long long)un * xd < (long long)xn * den) {
            xn = un;
            xd = den;
        }
    }
    return (long long)en * xd <= (long long)xn * ed;
}

struct TileSmem {
    int count;
    int item;
    int layer, tx, ty;
    int n_und;
    int pub[4];   // record, first chunk, chunks published, offset of the ids in the pool
};

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src)
{
    unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// True if the box [lo, hi] (target frame) certainly (margin > band) blocks
// the segments from q to all four extreme patch centres; see below.
__device__ __forceinline__ bool box_blocks_all(const DevRequest &R, float4 lo, float4 hi, float qu, float qn,
                                               float qw)
{
    const float du0 = R.u_min - qu, du1 = R.u_max - qu;
    const float dn = R.p_n - qn;
    const float dw0 = R.w_min - qw, dw1 = R.w_max - qw;
    const float iu0 = rcp_approx(du0), iu1 = rcp_approx(du1), inn = rcp_approx(dn);
    const float iw0 = rcp_approx(dw0), iw1 = rcp_approx(dw1);
    const float au = lo.x - qu, bu = hi.x - qu, an = lo.y - qn, bn = hi.y - qn;
    const float aw = lo.z - qw, bw = hi.z - qw;
    const float nu0 = (du0 >= 0.f ? au : bu) * iu0, fu0 = (du0 >= 0.f ? bu : au) * iu0;
    const float nu1 = (du1 >= 0.f ? au : bu) * iu1, fu1 = (du1 >= 0.f ? bu : au) * iu1;
    const float nw0 = (dw0 >= 0.f ? aw : bw) * iw0, fw0 = (dw0 >= 0.f ? bw : aw) * iw0;
    const float nw1 = (dw1 >= 0.f ? aw : bw) * iw1, fw1 = (dw1 >= 0.f ? bw : aw) * iw1;
    const float e0 = fmaxf((dn >= 0.f ? an : bn) * inn, 0.f);
    const float x0 = fminf((dn >= 0.f ? bn : an) * inn, 1.f);
    return fminf(fminf(fu0, fw0), x0) - fmaxf(fmaxf(nu0, nw0), e0) > kBand &&
           fminf(fminf(fu1, fw0), x0) - fmaxf(fmaxf(nu1, nw0), e0) > kBand &&
           fminf(fminf(fu0, fw1), x0) - fmaxf(fmaxf(nu0, nw1), e0) > kBand &&
           fminf(fminf(fu1, fw1), x0) - fmaxf(fmaxf(nu1, nw1), e0) > kBand;
}

// One-box check.  On the target plane the points whose segment to q meets a
// convex box form a convex set (a segment from q to any point between two
// blocked ones crosses the box between their two hit points), and every patch
// centre lies in the rectangle spanned by the extreme ones, so a box that
// blocks the four extreme patches blocks every patch.  Only margins above the
// band count, so the answer is exact.

// Does a viewpoint at normal coordinate qn see the measured side of the
// target?  One-sided: n.(q - p) > 0.  Two-sided: anywhere off its plane.
__device__ __forceinline__ bool facing(const DevRequest &R, float qn)
{
    return (R.flags & VCM_TWO_SIDED) ? qn != R.p_n : R.sn * (qn - R.p_n) > 0.f;
}

// Field-of-view cone (Section III-B, Table II): is q inside the cone of the
// patch at q - r, a.r >= c |r|?  r comes in target-frame components
// (u, n, w), each the rounded float difference q - p; the test runs in world
// order x, y, z with one float32 rounding per operation (no fused
// multiply-add), as the request header states, which errs in the margin by
// at most about 10.5 u |r|: only pairs within 1e-6 |r| of the cone's edge
// can be decided differently from the exact inequality.
__device__ __forceinline__ bool in_cone_inline(const DevRequest &R, float ru, float rn, float rw)
{
    const float r0 = R.au == 0 ? ru : (R.an == 0 ? rn : rw);
    const float r1 = R.au == 1 ? ru : (R.an == 1 ? rn : rw);
    const float r2 = R.au == 2 ? ru : (R.an == 2 ? rn : rw);
    float d = __fadd_rn(__fmul_rn(R.cone_a[0], r0), __fmul_rn(R.cone_a[1], r1));
    d = __fadd_rn(d, __fmul_rn(R.cone_a[2], r2));
    if (R.flags & VCM_TWO_SIDED)
        d = fabsf(d);
    float rr = __fadd_rn(__fmul_rn(r0, r0), __fmul_rn(r1, r1));
    rr = __fadd_rn(rr, __fmul_rn(r2, r2));
    return d >= __fmul_rn(R.cone_c, __fsqrt_rn(rr));
}

// All patches of the target at once: kConeIn if every one counts for the
// viewpoint, kConeOut if none does, kConeMixed if the patches have to be tested
// one by one.  Mostly one of the first two, for 40 operations instead of 25
// per patch.  With r = q - p and a margin of 1e-5 |r|, far above the test's 6.3e-7
// |r|, so that the classes agree with in_cone_inline:
//  * a.r - (c + 1e-5) |r| is concave in r for c >= -1e-5, so it is >= 0 on the
//    whole patch rectangle if it is at its four corners (a two-sided cone: for
//    one sign of a at all corners);
//  * it is at most a.r0 + rho - c |r0| + |c| rho around the centre r0 with half
//    diagonal rho.
// Called by whole warps with the same viewpoint.
enum { kConeOut = 0, kConeIn = 1, kConeMixed = 2 };
__device__ __forceinline__ int cone_class(const DevRequest &R, float qu, float qn, float qw)
{
    constexpr float kSlack = 1e-5f;
    const int lane = threadIdx.x & 31;
    const float a_u = R.cone_a[R.au], a_n = R.cone_a[R.an], a_w = R.dims == 3 ? R.cone_a[R.aw] : 0.f;
    const bool two = (R.flags & VCM_TWO_SIDED) != 0;
    const float rn = qn - R.p_n;
    {
        const float eu = 0.5f * (R.u_max - R.u_min), ew = 0.5f * (R.w_max - R.w_min);
        const float ru = qu - 0.5f * (R.u_min + R.u_max), rw = qw - 0.5f * (R.w_min + R.w_max);
        const float rho = 1.0001f * sqrtf(fmaf(eu, eu, ew * ew));
        const float len = sqrtf(fmaf(ru, ru, fmaf(rn, rn, rw * rw)));
        float d = fmaf(a_u, ru, fmaf(a_n, rn, a_w * rw));
        d = two ? fabsf(d) : d;
        if (d + rho - R.cone_c * len + fabsf(R.cone_c) * rho < -kSlack * (len + rho))
            return kConeOut;
    }
    if (R.cone_c < -kSlack)
        return kConeMixed;
    const float ru = qu - ((lane & 1) ? R.u_max : R.u_min), rw = qw - ((lane & 2) ? R.w_max : R.w_min);
    const float need = (R.cone_c + kSlack) * sqrtf(fmaf(ru, ru, fmaf(rn, rn, rw * rw)));
    const float d = fmaf(a_u, ru, fmaf(a_n, rn, a_w * rw));
    return __all_sync(kFull, d >= need) || (two && __all_sync(kFull, -d >= need)) ? kConeIn : kConeMixed;
}

// One patch's test, not inlined, for the sweep (keeps its code small).
__device__ __noinline__ bool in_cone(const DevRequest &R, float ru, float rn, float rw)
{
    return in_cone_inline(R, ru, rn, rw);
}

// One row of a column against a box, in float32 with the exact re-decision in
// the band: the segment q -> (pu, p_n, pw).  Bit 0: blocked, bit 1: re-decided.
// Not inlined: the sweep takes it for rows at the end of a box's interval only.
__device__ __noinline__ unsigned row_hit(float qu, float qn, float qw, float pu, float pn, float pw, float4 lo,
                                         float4 hi, bool is3d)
{
    const float du = pu - qu, dn = pn - qn, dw = pw - qw;
    const float iu = rcp_approx(du), in = rcp_approx(dn);
    float enter = fmaxf(fmaxf(((du >= 0.f ? lo.x : hi.x) - qu) * iu, ((dn >= 0.f ? lo.y : hi.y) - qn) * in), 0.f);
    float leave = fminf(fminf(((du >= 0.f ? hi.x : lo.x) - qu) * iu, ((dn >= 0.f ? hi.y : lo.y) - qn) * in), 1.f);
    if (is3d) {
        const float iw = rcp_approx(dw);
        enter = fmaxf(enter, ((dw >= 0.f ? lo.z : hi.z) - qw) * iw);
        leave = fminf(leave, ((dw >= 0.f ? hi.z : lo.z) - qw) * iw);
    }
    const float margin = leave - enter;
    if (margin > kBand)
        return 1u;
    if (margin < -kBand)
        return 0u;
    return 2u | (exact_hit(qu, qn, qw, pu, pn, pw, lo, hi) ? 1u : 0u);
}

// Bits [start, start + n) of a word; start 0..32, n 0..32.
__device__ __forceinline__ unsigned bit_run(int start, int n)
{
    unsigned m;
    asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(m) : "r"(start), "r"(n));
    return m;
}

// One viewpoint swept by one warp.  Lane l owns patch column cp * nuc +
// l % nuc and, of the pass's 32 x groups rows, the rows (rp * 32 + m) * groups
// + l / nuc, m < 32, one bit each.
//
// What bounded the sweep was instruction issue: one test per (row, box).  But
// the rows of a column that a box blocks are one interval.  The column's
// segment is inside the box's u and n slabs for t in [E, X]; it reaches the
// box's w extent [a, b] for some such t iff its w offset dw lies in
//     [a / (a > 0 ? X : E), b / (b > 0 ? E : X)],
// the union over t of [a / t, b / t].  So a box and a column take one interval
// in row numbers and one bit mask, about 40 lane operations for up to 32 rows
// where the row tests took 15 + 8 per row, and the lane holds no per-row state
// (16 registers), nor are there variants by rows per pass.
//
// Only the reciprocals 1/E and 1/X are needed.  Per (viewpoint, box) they come
// from reciprocals of the box's offsets, which one lane per box forms ahead
// (the record); per column they are products with du:
//     iE = min(du r_u + k_u, nE),  iX = max(du f1, du f2, nX).
// A box beside q in u (a_u > 0 or b_u < 0) has r_u = 1 / its near face and
// k_u = 0, so a column on the other side gets iE <= 0 and misses; a box that
// spans q has r_u = 0, k_u = inf (it is entered at t = 0).  f1 and f2 are the
// far faces for du > 0 and du < 0.  With the hardware reciprocal iE and iX err
// by at most 5 u, so iE > iX (1 + 1e-6) is a certain u/n hit and iE < iX (1 -
// 1e-6) a certain miss.  An end of the interval in row numbers errs by at most
// 12 u (|c| + 33) with c = -dw0 / step, plus twice the rows' rounding to the
// lattice: rows within eps = 2 dev / step + 2e-6 (|c| + 64) of an end, and
// every row of an uncertain u/n test, go to row_hit, which has the 1e-6 band
// and the exact re-decision.  A lane whose eps passes 1/4 row (rows a few
// lattice units apart) takes row_hit for all its open rows.
//
// The boxes are filtered once per viewpoint, one per lane: a box whose shadow
// on the target plane, [du_lo, du_hi] x [dw_lo, dw_hi], misses the patch
// rectangle takes no further part.  The one-box test of the kept boxes comes
// from the same record: a box that certainly blocks the four extreme patches
// blocks them all (the one-box check), and the viewpoint is decided.  A
// viewpoint keeps its records over its column passes when at most 32 boxes
// are left (nearly always: 1 to 5).  When there are more (filter_stop: 32, with
// more than two passes 32 for each), the filter ends there and each pass filters
// the list again, 32 boxes at a time, nearest first, until no
// row is open: where that many boxes lie before the target a few near ones
// usually close it, and in strict mode the first blocked row does.  Filtered to its
// end for the sake of the one-box test, such a list cost more than it saved: 512^2
// viewpoints in 2D, 100,000 rectangles of 0.3 to 1 m in 1 km, 330 -> 263 us, strict
// 310 -> 195; as posts, 256^2 x 2 viewpoints, 32 x 16 patches, 404 -> 315, strict
// 372 -> 195; of 0.5 to 3 m in 10 km 263 -> 292 (2D) and 327 -> 312 (posts).  Long
// lists without the filter are faster still where no box hides the viewpoint (281
// and 144 us for the posts), but in cities one further on often does: 100,000
// rectangles of 5 to 30 m in 10 km 99 us, without 158; with bits, 512^2 x 2
// viewpoints, 60 m target 306 and 441.  A hiding box behind 32 others is missed: 4.5
// M viewpoints, 100 m target, one scene 654 -> 680 us, another 1.63 -> 1.38 ms.
// The more passes, the more that costs: 16 of them (100 x 100 patches, strict, bits)
// 2.23 -> 2.97 ms, with 32 boxes per pass 2.32; 3 (31 x 65) 61 -> 84, 61.5 us.  Two
// (64 patches in 2D) are better with 32: the first of the scenes above 263 and 283 us.
//
// Measured against the row tests (both passes; 2,048^2 x 8 viewpoints, 100,000
// boxes, 64 x 32 patches: 10.9 -> 5.4 ms; 512^2 x 5, 5,000 boxes, 32 x 16:
// 0.247 -> 0.164 ms, with bits 0.41 -> 0.267; 64 uneven requests: 15.7 ->
// 8.9 ms).

constexpr float kLess = 1.f - 1e-6f, kMore = 1.f + 1e-6f;

// A rectangle of patch centres relative to a viewpoint, and the same widened
// by more than a shadow's rounding.
struct PatchRect {
    float u0, u1, w0, w1;          // smallest and largest offset along u and w
    float u_from, u_to, w_from, w_to;
};
__device__ __forceinline__ PatchRect patch_rect(float u0, float u1, float w0, float w1)
{
    const float su = 2e-6f * fmaxf(fabsf(u0), fabsf(u1)), sw = 2e-6f * fmaxf(fabsf(w0), fabsf(w1));
    return PatchRect{u0, u1, w0, w1, u0 - su, u1 + su, w0 - sw, w1 + sw};
}

// The record of one box for a viewpoint, if its shadow meets the rectangle:
// returns whether it does.  r0 = (r_u, k_u, f1, f2); r1 = (nE, nX, a, b) with a
// and b the w offsets whose quotients bound the rows from below and above (for
// rows that run down the w axis they trade places), in rows.
__device__ __forceinline__ bool make_record(float4 lo, float4 hi, float qu, float qn, float qw, float dn, bool is3d,
                                            float inv_row, const PatchRect &P, float4 &r0, float4 &r1)
{
    constexpr float kTiny = 1e-20f;   // stands for a zero offset: inf x kTiny = inf, and 0 otherwise
    const float a_u = lo.x - qu, b_u = hi.x - qu, a_n = lo.y - qn, b_n = hi.y - qn;
    // the n interval of every segment from q, as 1 / t
    const float D = fabsf(dn), N = dn >= 0.f ? a_n : -b_n, F = dn >= 0.f ? b_n : -a_n;
    const float nE = N > 0.f ? D * rcp_approx(N) : f_inf();
    const float nX = F > 0.f ? fmaxf(1.f, D * rcp_approx(F)) : D > 0.f ? f_inf() : 1.f;
    // offsets with the sign that the end's parameter depends on
    const float a_u1 = a_u > 0.f ? a_u : fminf(a_u, -kTiny), b_u1 = b_u < 0.f ? b_u : fmaxf(b_u, kTiny);
    bool keep = F >= 0.f && nE >= nX * kLess && a_u1 * (a_u > 0.f ? nX : nE) <= P.u_to &&
                b_u1 * (b_u < 0.f ? nX : nE) >= P.u_from;
    float a_w = -f_inf(), b_w = f_inf();   // unbounded in 2D
    if (is3d) {
        a_w = lo.z - qw;
        b_w = hi.z - qw;
        a_w = a_w > 0.f ? a_w : fminf(a_w, -kTiny);
        b_w = b_w < 0.f ? b_w : fmaxf(b_w, kTiny);
        keep = keep && a_w * (a_w > 0.f ? nX : nE) <= P.w_to && b_w * (b_w < 0.f ? nX : nE) >= P.w_from;
    }
    if (!keep)
        return false;
    const bool out = a_u > 0.f || b_u < 0.f;
    const float r_a = a_u != 0.f ? rcp_approx(a_u) : -f_inf(), r_b = b_u != 0.f ? rcp_approx(b_u) : f_inf();
    r0 = make_float4(out ? (a_u > 0.f ? r_a : r_b) : 0.f, out ? 0.f : f_inf(), b_u < 0.f ? r_a : r_b,
                     a_u > 0.f ? r_b : r_a);
    r1 = make_float4(nE, nX, (inv_row >= 0.f ? a_w : b_w) * inv_row, (inv_row >= 0.f ? b_w : a_w) * inv_row);
    return true;
}

// True if a recorded box certainly blocks all four corners of the rectangle.
// Along w the bound of the smaller offset's side is a / dw > 0 only with a > 0.
__device__ __forceinline__ bool record_blocks_rect(float4 r0, float4 r1, float inv_row, const PatchRect &P)
{
    const float e0 = fminf(fmaf(P.u0, r0.x, r0.y), r1.x), e1 = fminf(fmaf(P.u1, r0.x, r0.y), r1.x);
    const float x0 = fmaxf(fmaxf(P.u0 * r0.z, P.u0 * r0.w), r1.y), x1 = fmaxf(fmaxf(P.u1 * r0.z, P.u1 * r0.w), r1.y);
    // per column the w offsets it blocks for certain: (from, to), as in the sweep
    const float row = fabsf(inv_row), a = inv_row >= 0.f ? r1.z : -r1.w, b = inv_row >= 0.f ? r1.w : -r1.z;
    const float from = fmaxf(a * (a > 0.f ? x0 : e0), a * (a > 0.f ? x1 : e1));
    const float to = fminf(b * (b > 0.f ? e0 : x0), b * (b > 0.f ? e1 : x1));
    return e0 > x0 * kMore && e1 > x1 * kMore && from < P.w_from * row && to > P.w_to * row;
}

// The filter of one pass for a viewpoint with more than 32 kept boxes: lanes over
// the boxes [base, base + 32); returns the kept ones, records written.  Of boxes
// that block the whole pass one is enough.
__device__ __noinline__ unsigned pass_records(const DevRequest &R, const float4 *__restrict__ sbox, int n_smem,
                                              Tail spill, int count,
                                              const float4 *__restrict__ gbox, float qu, float qn, float qw, int cp,
                                              int row0, float4 *rec, int n_boxes, int base)
{
    const int lane = threadIdx.x & 31;
    const float ua = R.u_coord[cp * R.nuc] - qu, ub = R.u_coord[min(R.nu, cp * R.nuc + R.nuc) - 1] - qu;
    const float wa = R.w_coord[row0] - qw, wb = R.w_coord[min(R.nw, row0 + 32 * R.groups) - 1] - qw;
    const PatchRect P = patch_rect(fminf(ua, ub), fmaxf(ua, ub), fminf(wa, wb), fmaxf(wa, wb));
    bool keep = base + lane < count, full = false;
    if (keep) {
        float4 lo, hi, r0, r1;
        load_box(sbox, n_smem, spill, gbox, base + lane, n_boxes, R.stats, lo, hi);
        keep = make_record(lo, hi, qu, qn, qw, R.p_n - qn, R.dims == 3, R.inv_row, P, r0, r1);
        if (keep) {
            rec[2 * lane] = r0;
            rec[2 * lane + 1] = r1;
            full = record_blocks_rect(r0, r1, R.inv_row, P);
        }
    }
    const unsigned kept = __ballot_sync(kFull, keep), whole = __ballot_sync(kFull, full);
    return whole ? whole & (0u - whole) : kept;
}

// Where a lane stands in a request's patch grid, in one register: bits 0-12 its
// column of a pass (nu for the lanes past the last row group, which own none),
// 13-17 its row group, 18-30 that group's rows.
struct LaneMap {
    unsigned bits;
    __device__ __forceinline__ int c_in() const { return (int)(bits & 0x1fffu); }
    __device__ __forceinline__ int g() const { return (int)((bits >> 13) & 31u); }
    __device__ __forceinline__ int rows() const { return (int)(bits >> 18); }
};
__device__ __forceinline__ LaneMap lane_map(const DevRequest &R)
{
    const int lane = threadIdx.x & 31;
    int g = lane / R.nuc;
    const int c_in = g < R.groups ? lane - g * R.nuc : R.nu;
    g = min(g, R.groups - 1);
    return LaneMap{(unsigned)c_in | ((unsigned)g << 13) | ((unsigned)((R.nw - g + R.groups - 1) / R.groups) << 18)};
}
// Row groups are this far apart in a warp's staged rows; 0: they do not fit.
__device__ __forceinline__ int row_stride(const DevRequest &R)
{
    const int stride = (R.rows + 3) & ~3;
    return R.groups * stride <= kRowCap ? stride : 0;
}
// staged rows: row i = m * G + g at g * stride + m (a float division is exact for these sizes)
__device__ __forceinline__ int row_slot(int i, int G, int stride)
{
    const int m = G == 1 ? i : (int)(((float)i + 0.5f) / (float)G);
    return (i - m * G) * stride + m;
}
// Shared memory of one warp's sweeps.
struct WarpScratch {
    float4 rec[2 * 32];   // records of the boxes left to a viewpoint
    float rw[kRowCap];    // row offsets q_w - w, each lane group's rows side by side
    float rw_of;          // the q_w they are for (NaN: none); viewpoints of a layer share them
    int rec_id[32];       // the records' boxes
};

// One open patch's term of the visible measure.  |r|^2 is (ru^2 + rn^2) of the
// column + rw^2 of the row.
template <bool EXTRA, bool IS3D>
__device__ __forceinline__ float measure_term(const DevRequest &R, bool mixed, float col_d2, float m_s, float ru,
                                              float rn, float rw)
{
    const float d2 = fmaf(rw, rw, col_d2);
    float term;
    if (IS3D) {
        const float ir = rsqrt_normal(d2);
        term = m_s * (ir * ir * ir);   // A |r| cos(theta) / |r|^3
    } else {
        term = m_s / d2;               // len |r| cos(theta) / |r|^2
    }
    if (EXTRA && mixed && !in_cone(R, ru, rn, rw))
        term = 0.f;   // q is outside this patch's field of view
    return term;
}

// Returns the viewpoint's value, or -1 if one box blocks every patch.
template <bool EXTRA>
__device__ __forceinline__ float sweep_viewpoint(const DevRequest &R, const LaneMap &M,
                                                 const float4 *__restrict__ sbox, int n_smem,
                                                 Tail spill, int count,
                                                 const float4 *__restrict__ gbox, float qu, float qn,
                                                 float qw, bool front, long long vp, WarpScratch &W,
                                                 unsigned &tests, unsigned &corners, unsigned &rechecks,
                                                 int n_boxes)
{
    constexpr float kMagic = 12582912.f;   // 1.5 x 2^23: adding it rounds to an integer
    float4 *rec = W.rec;
    const int lane = threadIdx.x & 31;
    const int nuc = R.nuc, G = R.groups;
    const float dn = R.p_n - qn;
    const bool want_bits = (R.flags & VCM_EMIT_BITS) && R.bits_out;
    const bool is3d = R.dims == 3;
    // strict: any blocked patch zeroes the viewpoint, so the first one ends it
    const bool strict = (R.flags & VCM_STRICT) != 0;
    const bool strict_exit = strict && !want_bits;
    bool strict_fail = false;
    const float inv_row = R.inv_row;
    float sum = 0.f, comp = 0.f;
    const int cone = EXTRA && R.cone ? cone_class(R, qu, qn, qw) : kConeIn;

    // the boxes that can block a patch at all, and the one-box test of each, until
    // filter_stop are kept.  Lists of at most 8 boxes go without the test:
    // the tile's checks mostly had these boxes, and a box that blocks every patch
    // closes the rows at its first interval anyway (with the test 73.1 us on
    // 512^2 x 5 viewpoints and 5,000 boxes, 71.9 without)
    int n_rec = 0;
    {
        const PatchRect P = patch_rect(R.u_min - qu, R.u_max - qu, R.w_min - qw, R.w_max - qw);
        for (int base = 0; base < count; base += 32) {
            bool keep = base + lane < count, full = false;
            float4 r0, r1;
            if (keep) {
                float4 lo, hi;
                load_box(sbox, n_smem, spill, gbox, base + lane, n_boxes, R.stats, lo, hi);
                keep = make_record(lo, hi, qu, qn, qw, dn, is3d, inv_row, P, r0, r1);
                if (keep && count > 8)
                    full = record_blocks_rect(r0, r1, inv_row, P);
            }
            const unsigned kept = __ballot_sync(kFull, keep);
            if (kept == 0u)
                continue;
            corners += count > 8 ? 4 * __popc(kept) : 0;
            if (__any_sync(kFull, full))
                return -1.f;
            const int at = n_rec + __popc(kept & ((1u << lane) - 1u));
            if (keep && at < 32) {
                rec[2 * at] = r0;
                rec[2 * at + 1] = r1;
                W.rec_id[at] = base + lane;
            }
            n_rec += __popc(kept);
            if (n_rec > R.filter_stop)   // the passes filter the list
                break;
        }
        __syncwarp();   // the records are written
    }
    if (want_bits) {   // the passes below set bits in the viewpoint's cleared words
        for (int wd = lane; wd < R.words; wd += 32)
            put_word(R, vp * R.words + wd, 0u);
        __syncwarp();
    }

    for (int cp = 0; cp < R.col_passes && !(strict_exit && strict_fail); ++cp) {
        const int iu = cp * nuc + M.c_in();
        const bool col_ok = iu < R.nu;
        const float pu = R.u_coord[col_ok ? iu : 0];
        const float du = pu - qu;
        // A lane's terms are added plainly over each 8 of its rows (error
        // <= 7u of the group's total, the terms being >= 0), and the group
        // totals with Neumaier's compensation, so the bound holds for any
        // patch count.
        for (int r_at = 0; r_at < R.rows && !(strict_exit && strict_fail); r_at += 32) {
            const int row0 = r_at * G;                          // the pass's first row
            const int rows = min(R.rows - r_at, 32);            // its rows per lane
            const int mine = col_ok ? min(M.rows() - r_at, 32) : 0;
            const unsigned valid = bit_run(0, max(mine, 0));
            const float *__restrict__ w_row = R.w_coord + row0 + M.g();   // row m: w_row[m * G]
            unsigned alive = valid;
            if (n_rec > 0) {
                const float c = -((mine > 0 ? w_row[0] : R.w_min) - qw) * inv_row;
                const float eps = fmaf(2.f * R.row_dev, fabsf(inv_row), 2e-6f * (fabsf(c) + 64.f));
                const bool coarse = !(eps < 0.25f);
                const float near_half = 0.5f - eps;
                const bool fits = n_rec <= 32;
                for (int base = 0; base < (fits ? 1 : count); base += 32) {
                    unsigned todo;
                    if (fits) {
                        todo = bit_run(0, n_rec);
                    } else {
                        todo = pass_records(R, sbox, n_smem, spill, count, gbox, qu, qn, qw, cp, row0, rec, n_boxes,
                                            base);
                        __syncwarp();   // the records are written
                    }
                    bool done = false;
                    while (todo) {
                        const int j = __ffs(todo) - 1;
                        todo &= todo - 1;
                        const float4 ru = rec[2 * j], rw = rec[2 * j + 1];
                        const float iE = fminf(fmaf(du, ru.x, ru.y), rw.x);
                        const float iX = fmaxf(fmaxf(du * ru.z, du * ru.w), rw.y);
                        tests += alive != 0u;
                        unsigned hit = 0u, ask = 0u;   // rows blocked for certain, rows to decide one by one
                        if (alive != 0u && iE >= iX * kLess) {
                            // first row + 1/2 and last row - 1/2 of the interval
                            const float y = fminf(fmaxf(fmaf(rw.z > 0.f ? iX : iE, rw.z, c + 0.5f), 0.f), 32.f);
                            const float z = fminf(fmaxf(fmaf(rw.w > 0.f ? iE : iX, rw.w, c - 0.5f), -1.f), 31.f);
                            const float ry = y + kMagic, rz = z + kMagic;
                            if (!coarse && iE > iX * kMore) {
                                const int from = __float_as_int(ry) - __float_as_int(kMagic);
                                hit = bit_run(from, max(__float_as_int(rz) - __float_as_int(ry) + 1, 0));
                                if (fabsf(y - (ry - kMagic)) > near_half)   // the row at the lower end
                                    ask = 1u << (__float2int_rn(y - 0.5f) & 31);
                                if (fabsf(z - (rz - kMagic)) > near_half)   // the row at the upper end
                                    ask |= 1u << (__float2int_rn(z + 0.5f) & 31);
                            } else {
                                ask = kFull;
                            }
                            ask &= alive;
                            hit &= ~ask;
                        }
                        if (__any_sync(kFull, ask != 0u)) {   // rare
                            float4 lo, hi;
                            load_box(sbox, n_smem, spill, gbox, fits ? W.rec_id[j] : base + j, n_boxes, R.stats, lo,
                                     hi);
                            // a column with many such rows (it grazes the box): its rows over the
                            // lanes, where that takes fewer steps than every lane doing its own
                            // (28 x 8 patches, 73,000 viewpoints that many boxes graze in all
                            // columns: 257 us without the comparison, 111 with it)
                            unsigned columns = __ballot_sync(kFull, __popc(ask) > 2);
                            if (columns && __popc(columns) >= (int)__reduce_max_sync(kFull, (unsigned)__popc(ask)))
                                columns = 0u;
                            while (columns) {
                                const int from = __ffs(columns) - 1;
                                columns &= columns - 1;
                                const float p_col = __shfl_sync(kFull, pu, from);
                                const unsigned rows_of = __shfl_sync(kFull, ask, from);
                                const int g_of = __shfl_sync(kFull, M.g(), from);
                                unsigned h = 0u;
                                if ((rows_of >> lane) & 1u)
                                    h = row_hit(qu, qn, qw, p_col, R.p_n, R.w_coord[row0 + lane * G + g_of], lo, hi, is3d);
                                rechecks += h >> 1;
                                const unsigned blocked_rows = __ballot_sync(kFull, h & 1u);
                                if (lane == from) {
                                    hit |= blocked_rows;
                                    ask = 0u;
                                }
                            }
                            while (ask) {
                                const int m = __ffs(ask) - 1;
                                ask &= ask - 1;
                                const unsigned h = row_hit(qu, qn, qw, pu, R.p_n, w_row[m * G], lo, hi, is3d);
                                hit |= (h & 1u) << m;
                                rechecks += h >> 1;
                            }
                        }
                        alive &= ~hit;
                        if (__all_sync(kFull, alive == 0u) || (strict_exit && __any_sync(kFull, alive != valid))) {
                            done = true;
                            break;
                        }
                    }
                    __syncwarp();   // the records are read before others are written
                    if (done)
                        break;
                }
            }
            if (strict)
                strict_fail |= __any_sync(kFull, alive != valid);
            if (want_bits) {
                // The blocked bits.  Row m of the pass is one run of patches
                // over the lanes, from patch j0, so a ballot is its bits and
                // lane m adds them to the two words they fall into (bit by
                // bit atomics took a third of the 5,000-box step with bits).
                unsigned run = 0u;
                const unsigned blocked = valid & ~alive;
                for (int m = 0; m < rows; ++m) {
                    const unsigned b = __ballot_sync(kFull, (blocked >> m) & 1u);
                    if (lane == m)
                        run = b;
                }
                if (run) {
                    const int j0 = (row0 + lane * G) * R.nu + cp * nuc;
                    const long long at = vp * R.words + (j0 >> 5);
                    const unsigned first = run << (j0 & 31), rest = (j0 & 31) ? run >> (32 - (j0 & 31)) : 0u;
                    if (first && IN_BOUNDS(at, (long long)R.nx * R.ny * R.nl * R.words, R.stats))
                        atomicOr(&R.bits_out[at], first);
                    if (rest && IN_BOUNDS(at + 1, (long long)R.nx * R.ny * R.nl * R.words, R.stats))
                        atomicOr(&R.bits_out[at + 1], rest);
                }
            }
            // the visible measure of the open rows
            const unsigned open = front && !strict_fail && cone != kConeOut ? alive : 0u;
            if (!__any_sync(kFull, open != 0u))
                continue;
            const float ru = qu - pu, rn = qn - R.p_n;
            const float col_d2 = fmaf(ru, ru, rn * rn);
            // measure x |r| cos(theta); a two-sided target is measured from either side
            const float m_s = R.measure * ((EXTRA && (R.flags & VCM_TWO_SIDED)) ? fabsf(rn) : R.sn * rn);
            // Eight rows' terms in row order.  A closed row adds +0, which
            // changes nothing (the terms are >= 0), so the rows take no
            // branch; the add must not fuse with the term's product.  The
            // group total joins by a two-sum of the larger and the smaller
            // (both are >= 0).
            auto close_group = [&](float part) {
                const float tsum = sum + part;
                comp += (fmaxf(sum, part) - tsum) + fminf(sum, part);
                sum = tsum;
            };
            if (!is3d) {   // one row
                close_group(open & 1u ? measure_term<EXTRA, false>(R, cone == kConeMixed, col_d2, m_s, ru, rn, 0.f) : 0.f);
                continue;
            }
            const int stride = row_stride(R);
            if (stride > 0 && !(W.rw_of == qw)) {
                __syncwarp();   // the viewpoint before this one is done with them
                for (int i = lane; i < R.nw; i += 32)
                    W.rw[row_slot(i, G, stride)] = qw - R.w_coord[i];
                if (lane == 0)
                    W.rw_of = qw;
                __syncwarp();
            }
            const float *my_rw = W.rw + M.g() * stride + r_at;
            for (int m0 = 0; m0 < rows; m0 += 8) {
                const unsigned o8 = open >> m0;
                const unsigned any = __ballot_sync(kFull, (o8 & 0xffu) != 0u);
                if (any == 0u)
                    continue;
                float part = 0.f;
                if (stride > 0 && m0 + 8 <= rows) {
                    float t8[8];
                    if (EXTRA && cone == kConeMixed) {
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            t8[k] = measure_term<EXTRA, true>(R, true, col_d2, m_s, ru, rn, my_rw[m0 + k]);
                    } else {
                        // measure_term two rows at a time: the sweep is bound by issue
                        const ulonglong2 *s2 = reinterpret_cast<const ulonglong2 *>(my_rw + m0);
                        const ulonglong2 wa = s2[0], wb = s2[1];
                        const f32x2 w2[4] = {wa.x, wa.y, wb.x, wb.y}, c2 = pack2(col_d2, col_d2), m2 = pack2(m_s, m_s);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float d0, d1;
                            unpack2(fma2(w2[k], w2[k], c2), d0, d1);
                            const f32x2 ir = pack2(rsqrt_normal(d0), rsqrt_normal(d1));
                            unpack2(mul2(m2, mul2(mul2(ir, ir), ir)), t8[2 * k], t8[2 * k + 1]);
                        }
                    }
                    if (__all_sync(kFull, (o8 & 0xffu) == 0xffu)) {   // mostly
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            part = __fadd_rn(part, t8[k]);
                    } else {
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            part = __fadd_rn(part, (o8 & (1u << k)) ? t8[k] : 0.f);
                    }
                } else {
                    for (int m = m0; m < min(m0 + 8, rows); ++m) {
                        const bool counts = (open >> m) & 1u;
                        const float rw = stride > 0 ? my_rw[m] : counts ? qw - w_row[m * G] : 0.f;
                        const float t = measure_term<EXTRA, true>(R, cone == kConeMixed, col_d2, m_s, ru, rn, rw);
                        part = __fadd_rn(part, counts ? t : 0.f);
                    }
                }
                close_group(part);
            }
        }
    }
    float v = sum + comp;
    // fixed-order butterfly: every lane ends with the same value
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        v += __shfl_xor_sync(kFull, v, off);
    return strict_fail ? 0.f : v;
}

// A viewpoint in the target frame.
__device__ __forceinline__ float3 in_target_frame(const DevRequest &R, float qx, float qy, float zq)
{
    return make_float3(R.au == 0 ? qx : (R.au == 1 ? qy : zq), R.an == 0 ? qx : (R.an == 1 ? qy : zq),
                       R.dims == 3 ? (R.aw == 0 ? qx : (R.aw == 1 ? qy : zq)) : 0.f);
}

// One open viewpoint q: swept, and its outputs written.  Returns its value.
template <bool EXTRA>
__device__ __forceinline__ float sweep_one(const DevRequest &R, const LaneMap &M, float3 q, bool front, long long vp,
                                           const float4 *__restrict__ sbox, int n_smem, Tail tail, int count,
                                           const float4 *__restrict__ gbox, WarpScratch &W, unsigned &tests,
                                           unsigned &corners, unsigned &rechecks, unsigned &shortcuts, int n_boxes)
{
    const int lane = threadIdx.x & 31;
    float v = sweep_viewpoint<EXTRA>(R, M, sbox, n_smem, tail, count, gbox, q.x, q.y, q.z, front, vp, W, tests,
                                     corners, rechecks, n_boxes);
    if (v < 0.f) {   // one box blocks every patch
        ++shortcuts;
        if ((R.flags & VCM_EMIT_BITS) && R.bits_out)
            for (int wd = lane; wd < R.words; wd += 32) {
                const int rem = R.P - 32 * wd;
                put_word(R, vp * R.words + wd, rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u));
            }
    }
    v = front ? fmaxf(v, 0.f) : 0.f;
    if (lane == 0)
        put_v(R, vp, v);
    return v;
}

// Viewer-centric cell (VCM_VIEWER): one segment from the cell q to the
// viewer p (world frame) against the candidate boxes, nearest first; the
// cell's value is the visual angle (2D, Eq. 1) or solid angle (3D) of an
// object of size S at distance D facing the viewer, 0 when blocked or D = 0.
__device__ __forceinline__ float viewer_cell(const DevRequest &R, const float4 *__restrict__ sbox, int n_smem,
                                             Tail spill, int count,
                                             const float4 *__restrict__ gbox, float qx, float qy, float qz,
                                             bool &blocked, unsigned long long &tests, unsigned &rechecks,
                                             int n_boxes)
{
    const float px = R.u_min, py = R.p_n, pz = R.w_min;
    const float dx = px - qx, dy = py - qy, dz = pz - qz;
    const float ix = rcp_approx(dx), iy = rcp_approx(dy), iz = rcp_approx(dz);
    blocked = false;
    for (int i = 0; i < count && !blocked; ++i) {
        float4 lo, hi;
        load_box(sbox, n_smem, spill, gbox, i, n_boxes, R.stats, lo, hi);
        ++tests;
        const float ax = lo.x - qx, bx = hi.x - qx, ay = lo.y - qy, by = hi.y - qy, az = lo.z - qz, bz = hi.z - qz;
        const float enter = fmaxf(fmaxf((dx >= 0.f ? ax : bx) * ix, (dy >= 0.f ? ay : by) * iy),
                                  fmaxf((dz >= 0.f ? az : bz) * iz, 0.f));
        const float exit_ = fminf(fminf((dx >= 0.f ? bx : ax) * ix, (dy >= 0.f ? by : ay) * iy),
                                  fminf((dz >= 0.f ? bz : az) * iz, 1.f));
        const float mv = exit_ - enter;
        if (mv >= -kBand) {
            blocked = mv > kBand;
            if (!blocked) {
                ++rechecks;
                blocked = exact_hit(qx, qy, qz, px, py, pz, lo, hi);
            }
        }
    }
    const float D = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    if (blocked || !(D > 0.f))
        return 0.f;
    const float S = R.measure;
    if (R.dims == 2)
        return 2.f * atanf(S / (2.f * D));
    return 4.f * asinf(S * S / fmaf(4.f * D, D, S * S));
}


// If a box may matter to the tile, add it to the tile's candidate list (shared
// memory, then the block's spill region).
__device__ __forceinline__ void add_candidate(const float4 *__restrict__ world, const Swept &hull, int s,
                                              TileSmem &sm, int *s_ids, int list_cap, Tail spill,
                                              int spill_slot, const DevRequest &R, int n_boxes)
{
    if (!swept_meets(hull, world[2 * s], world[2 * s + 1]))
        return;
    const int pos = atomicAdd(&sm.count, 1);
    if (pos < list_cap)
        s_ids[pos] = s;
    else if (spill_slot >= 0) {
        if (IN_BOUNDS(pos - list_cap, n_boxes, R.stats))
            spill.put(pos - list_cap, s);
    } else {
        R.stats->error = VCM_DEVERR_SPILL_WAIT;   // no spill region: the result is flagged
    }
}

// Shared memory of the tile pass that its phases use in turn: the walk over the
// grid cells and the sort, the viewpoints to check, then (rarely) the sweeps of
// sweep_kept.
union TileScratch {
    struct {
        int rowpre[kThreads], rowx[kThreads], wsum[kWarps];   // cell-row spans
        int passb[kPassCap], passn[kPassCap], passp[kPassCap + 1], wsum2[kWarps];   // listed cells
        int hist[kDistClasses];   // counting sort of long candidate lists
    } walk;
    unsigned short check[kMaxTileViewpoints];   // viewpoints to check one by one
    WarpScratch sweep[kKeptWarps];
};

// The open viewpoints that a tile does not publish (no second pass, a full arena in
// the last round, a list past the arena), swept by the tile's first warps.  Not
// inlined: the tile pass then holds none of the sweep's registers.
__device__ __noinline__ void sweep_kept(const DevRequest &R, TileScratch &T, const float4 *__restrict__ sbox,
                                        int n_smem, Tail spill, int count,
                                        const float4 *__restrict__ gbox, const unsigned short *und, int *next,
                                        int n_und, int ix0, int iy0, int layer, int n_boxes)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= kKeptWarps)
        return;
    const LaneMap M = lane_map(R);
    const float zq = R.z_coord[layer];
    if (lane == 0)
        T.sweep[warp].rw_of = __int_as_float(0x7fffffff);
    __syncwarp();
    unsigned long long tests = 0, corners = 0;
    unsigned rechecks = 0, shortcuts = 0;
    float vmax = 0.f;
    for (;;) {
        int k = 0;
        if (lane == 0)
            k = atomicAdd(next, 1);
        k = __shfl_sync(kFull, k, 0);
        if (k >= n_und)
            break;
        unsigned vp_tests = 0, vp_corners = 0;
        const int ix = ix0 + (und[k] & 255), iy = iy0 + (und[k] >> 8);
        const float3 q = in_target_frame(R, R.x_coord[ix], R.y_coord[iy], zq);
        const float v = sweep_one<true>(R, M, q, facing(R, q.y), ((long long)layer * R.ny + iy) * R.nx + ix, sbox, n_smem,
                                        spill, count, gbox, T.sweep[warp], vp_tests, vp_corners, rechecks, shortcuts,
                                        n_boxes);
        vmax = fmaxf(vmax, v);
        tests += vp_tests;
        corners += vp_corners;
    }
    rechecks = __reduce_add_sync(kFull, rechecks);
    for (int off = 16; off > 0; off >>= 1)
        tests += __shfl_xor_sync(kFull, tests, off);
    if (lane == 0) {
        atomicMax(&R.stats->vmax_bits, __float_as_uint(vmax));
        atomicAdd(&R.stats->slab_tests, tests);
        atomicAdd(&R.stats->corner_tests, corners);
        if (shortcuts)
            atomicAdd(&R.stats->shortcut_viewpoints, (unsigned long long)shortcuts);
        if (rechecks)
            atomicAdd(&R.stats->rechecked, (unsigned long long)rechecks);
    }
}

// TILE_CHECK: the instantiation that looks at recorded blockers before a tile's
// cull (kTileCheckMinPatches).
//
// The pass holds no sweep: every viewpoint its checks leave open goes to the
// second pass (sweep_kept takes what does not fit).  It waits on latency (queue
// and cell loads, block barriers), so blocks per SM decide: 8 at 64 registers,
// where the sweep's registers allowed 6.  2,048^2 x 8 viewpoints, 100,000 boxes:
// 1.91 -> 1.47 ms for this pass; 512^2 x 5, 5,000 boxes 72 -> 61 us.  With 7 and 6
// blocks 1.57 and 1.72 ms; 9 blocks (56 registers) spill, 2 % slower.
template <bool TILE_CHECK>
__global__ void __launch_bounds__(kThreads, kTileBlocks)
k_tiles(DevScene sc, const DevRequest *__restrict__ reqs, const int *__restrict__ tile_prefix,
        int n_req, int total_tiles, int *__restrict__ work, Arena ar, unsigned char *__restrict__ spill_all, int id_bytes, int box_cap,
        int list_cap, int one_tile, int *__restrict__ spill_busy, int spill_slots, int share, int claim_rounds, int stop_at,
        int round)
{
    after_previous_kernel();
    if (round > 0 && __syncthreads_or(__ldcg(work) >= total_tiles))
        return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *s_box = reinterpret_cast<float4 *>(smem_raw);
    int *s_ids = reinterpret_cast<int *>(smem_raw + (size_t)box_cap * 32);
    __shared__ TileSmem sm;
    __shared__ float s_A[3][2], s_B[3][2];   // the tile's viewpoints and the target's patch rectangle: world axis, low and high
    __shared__ DevRequest s_req;
    __shared__ int s_next;             // viewpoints to check one by one
    __shared__ unsigned s_node[2][16];   // nodes' boxes, of this batch and the last
    __shared__ __align__(16) TileScratch s_scratch;
    __shared__ int s_req_idx, s_npass;
    __shared__ unsigned long long s_listed, s_shared;   // counters of thread 0
    __shared__ int s_next2;                     // cursor of the undecided list
    __shared__ unsigned short s_und[kMaxTileViewpoints];   // viewpoints left by the one-box check, x + 256 y
    auto &walk = s_scratch.walk;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    __shared__ int s_spill_slot;
    __shared__ bool s_full;   // the arena is nearly full: the block leaves its other tiles to the next round
    if (tid == 0) {
        s_full = false;
        s_req_idx = -1;
        s_npass = 0;
        s_listed = s_shared = 0;
        sm.item = -1;
        // A persistent block owns spill region blockIdx.x.  A one-tile block
        // claims a free region for the length of its tile.  There are as
        // many regions as blocks fit on the GPU, so a probe normally succeeds
        // at once; if every region is held (blocks of a preempted launch keep
        // theirs), it probes again after a pause, at most claim_rounds times
        // (kClaimRounds by default: a few ms), and then runs without one and
        // flags the result.
        int slot = (int)blockIdx.x;
        if (one_tile) {
            slot = -1;
            const int start = (int)(blockIdx.x % (unsigned)spill_slots);
            for (int round = 0; round < claim_rounds && slot < 0; ++round) {
                for (int probe = 0; probe < spill_slots && slot < 0; ++probe) {
                    const int c = (start + probe) % spill_slots;
                    if (atomicCAS(&spill_busy[c], 0, 1) == 0)
                        slot = c;
                }
                if (slot < 0)
                    __nanosleep(2000);
            }
        }
        s_spill_slot = slot;
    }
    __syncthreads();
    const int spill_slot = s_spill_slot;
    const Tail spill{spill_all + (size_t)max(spill_slot, 0) * spill_region_bytes(sc.n_boxes, id_bytes), id_bytes};
    // candidates past the staged boxes: ids in shared memory where these hold
    // every box of the scene (list_cap > box_cap), else the spill region
    const Tail tail = list_cap > box_cap ? Tail{s_ids + box_cap, 4} : spill;
    // counters, added to a request's when its last tile in a row is done
    vcm_stats *acc = nullptr;
    unsigned corner_tests = 0, shortcuts = 0;
    auto flush = [&] {
        corner_tests = __reduce_add_sync(kFull, corner_tests);
        shortcuts = __reduce_add_sync(kFull, shortcuts);
        if (acc && lane == 0) {
            if (corner_tests)
                atomicAdd(&acc->corner_tests, (unsigned long long)corner_tests);
            if (shortcuts)
                atomicAdd(&acc->shortcut_viewpoints, (unsigned long long)shortcuts);
        }
        if (acc && tid == 0) {
            atomicAdd(&acc->boxes_listed, s_listed);
            if (s_shared)
                atomicAdd(&acc->shared_viewpoints, s_shared);
            s_listed = s_shared = 0;
        }
        corner_tests = shortcuts = 0;
    };

    for (;;) {
        // thread 0 takes the next tile, copies its request and lays out the
        // two rectangles of the cull (one barrier for all of it).  With one_tile, block b
        // does tile b only and exits, so blocks of concurrent launches
        // interleave (a persistent grid would hold every SM to the end).
        if (tid == 0) {
            int it = s_full || (one_tile && sm.item == -2) ? total_tiles
                     : one_tile ? (int)blockIdx.x : atomicAdd(work, 1);
            // Queue order: last tile first, and within a request the
            // layers interleaved (consecutive items are one tile position
            // in every layer).  Measured on the 3D workload with the
            // target facing each of +-x and +-y: 3-14 % faster than the
            // plain order, never slower; either change alone was not.
            it = it < total_tiles ? total_tiles - 1 - it : total_tiles;
            sm.item = it;
            if (it < total_tiles) {
                // request of this tile: last r with tile_prefix[r] <= it
                int lo_r = 0, hi_r = n_req - 1;
                while (lo_r < hi_r) {
                    const int mid = (lo_r + hi_r + 1) >> 1;
                    if (tile_prefix[mid] <= it)
                        lo_r = mid;
                    else
                        hi_r = mid - 1;
                }
                if (lo_r != s_req_idx) {   // consecutive tiles mostly share a request
                    s_req = reqs[lo_r];
                    s_req_idx = lo_r;
                }
                const DevRequest &Q = s_req;
                // tile index within its request, layers interleaved
                const int t0 = it - tile_prefix[lo_r], pos = t0 / Q.nl, ly = t0 - pos * Q.nl;
                const int ty0 = pos / Q.tiles_x, tx0 = pos - ty0 * Q.tiles_x;
                sm.layer = ly;
                sm.tx = tx0;
                sm.ty = ty0;
                const int x0 = tx0 * Q.tile_x, x1 = min(Q.nx, x0 + Q.tile_x) - 1;
                const int y0 = ty0 * Q.tile_y, y1 = min(Q.ny, y0 + Q.tile_y) - 1;
                const float z = Q.z_coord[ly];
                sm.count = 0;
                sm.n_und = 0;
                s_next = 0;
                s_next2 = 0;
                s_A[0][0] = Q.x_coord[x0];
                s_A[0][1] = Q.x_coord[x1];
                s_A[1][0] = Q.y_coord[y0];
                s_A[1][1] = Q.y_coord[y1];
                s_A[2][0] = s_A[2][1] = Q.dims == 3 ? z : 0.f;
                s_B[Q.au][0] = Q.u_min;
                s_B[Q.au][1] = Q.u_max;
                s_B[Q.an][0] = s_B[Q.an][1] = Q.p_n;
                s_B[Q.aw][0] = Q.w_min;   // 0 in 2D
                s_B[Q.aw][1] = Q.w_max;
            }
        }
        __syncthreads();
        const int item = sm.item;
        if (item >= total_tiles)
            break;
        if (s_req.stats != acc) {
            flush();
            acc = s_req.stats;
        }
        const DevRequest &R = s_req;
        const int layer = sm.layer, tx = sm.tx, ty = sm.ty;
        const int ix0 = tx * R.tile_x, ix1 = min(R.nx, ix0 + R.tile_x);
        const int iy0 = ty * R.tile_y, iy1 = min(R.ny, iy0 + R.tile_y);
        const int tw = ix1 - ix0, tn = tw * (iy1 - iy0);
        // row of a tile index vi < 1024 in a row of tw <= 256: the float
        // product is within 1e-6 of vi / tw, whose fraction is 0.5 / tw away
        // from an integer, so the truncation is exact (and cheaper than an
        // integer division)
        const float inv_tw = 1.0f / (float)tw;
        const float zq = R.z_coord[layer];
        const bool want_bits = (R.flags & VCM_EMIT_BITS) && R.bits_out;

        // side of the target plane: s = sn (q_n - p_n) depends on q_n only
        float qn_lo, qn_hi;
        if (R.an == 2) {
            qn_lo = qn_hi = zq;
        } else if (R.an == 0) {
            qn_lo = R.x_coord[ix0]; qn_hi = R.x_coord[ix1 - 1];
        } else {
            qn_lo = R.y_coord[iy0]; qn_hi = R.y_coord[iy1 - 1];
        }
        const bool viewer = (R.flags & VCM_VIEWER) != 0;
        const bool any_front = viewer || (R.flags & VCM_TWO_SIDED) ||
                               (R.sn > 0.f ? (qn_hi - R.p_n > 0.f) : (R.p_n - qn_lo > 0.f));
        if (!any_front && !want_bits) {
            for (int i = tid; i < tn; i += kThreads) {
                const int ix = ix0 + i % tw, iy = iy0 + i / tw;
                put_v(R, ((long long)layer * R.ny + iy) * R.nx + ix, 0.f);
            }
            __syncthreads();
            if (tid == 0)
                sm.item = -2;
            continue;
        }

        // Shortcut from recorded blockers: a box that blocked this tile position on
        // another layer, or a neighbouring position, often blocks this tile
        // too, so 20 lanes test five of those first, each against the four extreme
        // patches from one of the tile's four corners; a tile one of them blocks
        // skips its cull.  Any tile writes the table, so which blocker it keeps is a
        // race; a box counts only if it certainly blocks, so results do not
        // depend on the table.
        bool pre_blocked = false;
        unsigned pre_tests = 0;
        if (TILE_CHECK && !viewer && R.blk_base >= 0) {
            int *blockers = work + kWorkHeader + ar.blocker_off();
            const int tile_pos = ty * R.tiles_x + tx;
            bool full = false;
            if (warp == 0) {
                // lanes 4c + k: candidate c (this position, then its four
                // neighbours) against corner viewpoint k of the tile
                const int c = lane >> 2, corner = lane & 3;
                int cand = -1;
                bool ok = false;
                if (c < 5) {
                    const int px = tx + (c == 1) - (c == 2), py = ty + (c == 3) - (c == 4);
                    cand = (px >= 0 && px < R.tiles_x && py >= 0 && py < R.tiles_y)
                               ? __ldcg(blockers + R.blk_base + py * R.tiles_x + px)
                               : -1;
                    if (cand >= 0 && cand < sc.n_boxes) {
                        const float4 *gb = sc.boxes[R.perm];
                        // the tile's corners from shared memory at each use, so that
                        // they are not held in registers through the cull
                        const float qx = s_A[0][corner & 1];
                        const float qy = s_A[1][corner >> 1];
                        const float qu = R.au == 0 ? qx : (R.au == 1 ? qy : zq);
                        const float qn = R.an == 0 ? qx : (R.an == 1 ? qy : zq);
                        const float qw = R.dims == 3 ? (R.aw == 0 ? qx : (R.aw == 1 ? qy : zq)) : 0.f;
                        ok = box_blocks_all(R, __ldg(&gb[2 * cand]), __ldg(&gb[2 * cand + 1]), qu, qn, qw);
                        pre_tests = 4;
                    }
                }
                const unsigned m = __ballot_sync(kFull, ok);
                full = c < 5 && ((m >> (4 * c)) & 0xFu) == 0xFu;
                if (full && corner == 0 && c != 0)
                    blockers[R.blk_base + tile_pos] = cand;
            }
            pre_blocked = __syncthreads_or(full) != 0;
        }

        // walk the grid cells under the hull's footprint.  In the xy plane
        // the footprint is the convex hull of two axis-aligned rectangles,
        // A (the tile's viewpoints) and B (the target's shadow on the
        // ground plane), which is the union over l in [0, 1] of the
        // rectangles (1 - l) A + l B.  A row of cells meets it for the l whose
        // rectangle reaches the row -- an interval, from two linear
        // inequalities -- and over the x-range those rectangles sweep, which
        // is spanned by the interval's two ends.  Rows are taken 128 at a
        // time: one thread finds a row's span, a block scan lays the spans
        // end to end, and the threads share out the cells.
        if (!pre_blocked) {
            const float ax0 = s_A[0][0], ax1 = s_A[0][1], ay0 = s_A[1][0], ay1 = s_A[1][1];
            const float bx0 = s_B[0][0], bx1 = s_B[0][1], by0 = s_B[1][0], by1 = s_B[1][1];
            const Swept hull = make_swept(s_A, s_B);
            // how far a cell's boxes reach past the cell, plus 1 m: far more
            // than the rounding of any quantity below (coordinates are
            // within 2^14 m), so no cell that can hold an occluder is missed
            const float oh = sc.overhang + 1.f;
            const int cy0 = max((int)floorf((fminf(ay0, by0) - oh - sc.gy0) * sc.inv_cell), 0);
            const int cy1 = min((int)floorf((fmaxf(ay1, by1) + oh - sc.gy0) * sc.inv_cell), sc.gny - 1);
            const float dy0 = by0 - ay0, dy1 = by1 - ay1;
            const float4 *world = sc.boxes[0];
            for (int r0 = cy0; r0 <= cy1; r0 += kThreads) {
                const int row = r0 + tid;
                int xa = 0, width = 0;
                if (row <= cy1) {
                    const float ya = fmaf((float)row, sc.cell, sc.gy0) - oh, yb = ya + sc.cell + 2.f * oh;
                    float l0 = 0.f, l1 = 1.f;
                    // lower edge ay0 + l dy0 <= yb
                    if (dy0 > 0.f)
                        l1 = fminf(l1, (yb - ay0) / dy0);
                    else if (dy0 < 0.f)
                        l0 = fmaxf(l0, (yb - ay0) / dy0);
                    else if (ay0 > yb)
                        l1 = -1.f;
                    // upper edge ay1 + l dy1 >= ya
                    if (dy1 > 0.f)
                        l0 = fmaxf(l0, (ya - ay1) / dy1);
                    else if (dy1 < 0.f)
                        l1 = fminf(l1, (ya - ay1) / dy1);
                    else if (ay1 < ya)
                        l1 = -1.f;
                    if (l0 <= l1) {
                        const float xl = fminf(fmaf(l0, bx0 - ax0, ax0), fmaf(l1, bx0 - ax0, ax0));
                        const float xh = fmaxf(fmaf(l0, bx1 - ax1, ax1), fmaf(l1, bx1 - ax1, ax1));
                        const int c0 = max((int)floorf((xl - oh - sc.gx0) * sc.inv_cell), 0);
                        const int c1 = min((int)floorf((xh + oh - sc.gx0) * sc.inv_cell), sc.gnx - 1);
                        if (c1 >= c0) {
                            xa = c0;
                            width = c1 - c0 + 1;
                        }
                    }
                }
                // exclusive scan of the widths over the block
                int incl = width;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, off);
                    if (lane >= off)
                        incl += t;
                }
                if (lane == 31)
                    walk.wsum[warp] = incl;
                __syncthreads();
                int before = 0, total = 0;
#pragma unroll
                for (int w2 = 0; w2 < kWarps; ++w2) {
                    before += w2 < warp ? walk.wsum[w2] : 0;
                    total += walk.wsum[w2];
                }
                walk.rowpre[tid] = before + incl - width;
                walk.rowx[tid] = xa;
                __syncthreads();
                // (a) threads over cells: the cells whose bounds meet the
                // hull are listed (box range start and length)
                for (int c = tid; c < total; c += kThreads) {
                    // the row of cell c: the last t with walk.rowpre[t] <= c
                    int t = 0;
#pragma unroll
                    for (int step = kThreads / 2; step > 0; step >>= 1)
                        if (walk.rowpre[t + step] <= c)
                            t += step;
                    const int cell = (r0 + t) * sc.gnx + walk.rowx[t] + (c - walk.rowpre[t]);
                    const int b = sc.cell_start[cell], e = sc.cell_start[cell + 1];
                    if (b == e || !swept_meets(hull, sc.cell_lo[cell], sc.cell_hi[cell]))
                        continue;
                    const int k = atomicAdd(&s_npass, 1);
                    if (k < kPassCap) {
                        walk.passb[k] = b;
                        walk.passn[k] = e - b;
                        continue;
                    }
                    for (int s = b; s < e; ++s)   // list full: this cell's boxes here
                        add_candidate(world, hull, s, sm, s_ids, list_cap, spill, spill_slot, R, sc.n_boxes);
                }
                __syncthreads();
                // (b) exclusive scan of the listed cells' box counts
                const int n_pass = min(s_npass, kPassCap);
                {
                    int cnt[kPassCap / kThreads], local = 0;
#pragma unroll
                    for (int q = 0; q < kPassCap / kThreads; ++q) {
                        const int k = tid * (kPassCap / kThreads) + q;
                        cnt[q] = k < n_pass ? walk.passn[k] : 0;
                        local += cnt[q];
                    }
                    int incl = local;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int t = __shfl_up_sync(kFull, incl, off);
                        if (lane >= off)
                            incl += t;
                    }
                    if (lane == 31)
                        walk.wsum2[warp] = incl;
                    __syncthreads();
                    int run = 0, all = 0;
#pragma unroll
                    for (int w2 = 0; w2 < kWarps; ++w2) {
                        run += w2 < warp ? walk.wsum2[w2] : 0;
                        all += walk.wsum2[w2];
                    }
                    run += incl - local;
#pragma unroll
                    for (int q = 0; q < kPassCap / kThreads; ++q) {
                        const int k = tid * (kPassCap / kThreads) + q;
                        walk.passp[k] = k < n_pass ? run : INT_MAX;
                        run += cnt[q];
                    }
                    if (tid == 0)
                        walk.passp[kPassCap] = all;
                }
                __syncthreads();
                // (c) threads over the listed cells' boxes
                const int n_boxes_listed = walk.passp[kPassCap];
                for (int i = tid; i < n_boxes_listed; i += kThreads) {
                    // the cell of box i: the last k with walk.passp[k] <= i
                    int k = 0;
#pragma unroll
                    for (int step = kPassCap / 2; step > 0; step >>= 1)
                        if (walk.passp[k + step] <= i)
                            k += step;
                    add_candidate(world, hull, walk.passb[k] + (i - walk.passp[k]), sm, s_ids, list_cap, spill, spill_slot, R,
                                  sc.n_boxes);
                }
                if (tid == 0)
                    s_npass = 0;
                __syncthreads();   // the next rows reuse the span arrays
            }
        }
        __syncthreads();
        // A block without a spill region (its bounded claim gave up) keeps
        // only the candidates it staged: its request is already flagged
        // (vcm_stats.error), and it reads no region it does not own.
        const int count = spill_slot >= 0 ? sm.count : min(sm.count, list_cap);
        const int n_smem = min(count, box_cap);
        const float4 *gbox = sc.boxes[R.perm];
        // near-first order of the staged candidates: nearby boxes block the
        // most sightlines, so the all-blocked exits come early.  Keys are the
        // squared footprint distance from the tile centre (a positive float,
        // so its bits order like the value) above the sorted box index.
        if (n_smem > 1) {
            const float cx = 0.5f * (R.x_coord[ix0] + R.x_coord[ix1 - 1]);
            const float cy = 0.5f * (R.y_coord[iy0] + R.y_coord[iy1 - 1]);
            auto key_of = [&](int i) {
                const int s = s_ids[i];
                const float4 l = world_box_lo(sc, s), h = world_box_hi(sc, s);
                const float dx = 0.5f * (l.x + h.x) - cx, dy = 0.5f * (l.y + h.y) - cy;
                return ((unsigned long long)__float_as_uint(fmaf(dx, dx, dy * dy)) << 32) | (unsigned)s;
            };
            if (n_smem <= 32) {
                // one warp, in registers
                if (warp == 0) {
                    unsigned long long key = lane < n_smem ? key_of(lane) : ~0ull;
#pragma unroll
                    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
                        for (int j = k >> 1; j > 0; j >>= 1) {
                            const unsigned long long other = __shfl_xor_sync(kFull, key, j);
                            const bool keep_min = ((lane & k) == 0) == ((lane & j) == 0);
                            key = keep_min ? (key < other ? key : other) : (key > other ? key : other);
                        }
                    if (lane < n_smem)
                        s_ids[lane] = (int)(key & 0xffffffffu);
                }
            } else {
                // longer lists: a counting sort into distance classes (4 per
                // doubling of the squared distance, 128 classes from 1 m^2),
                // near classes first; order within a class is arbitrary.
                // Results do not depend on the order, only how soon the
                // sweeps stop; this takes 4 barriers where a bitonic sort of
                // 256 keys took 36.
                int *cls_rank = reinterpret_cast<int *>(s_box);   // s_box is free until staging
                int *placed = cls_rank + n_smem;
                for (int i = tid; i < kDistClasses; i += kThreads)
                    walk.hist[i] = 0;
                __syncthreads();
                for (int i = tid; i < n_smem; i += kThreads) {
                    const unsigned bits = (unsigned)(key_of(i) >> 32);   // float bits of d^2 >= 0
                    const int c = (int)min((unsigned)(kDistClasses - 1), bits > 0x3f800000u ? (bits - 0x3f800000u) >> 21 : 0u);
                    cls_rank[i] = (c << 24) | atomicAdd(&walk.hist[c], 1);
                }
                __syncthreads();
                if (warp == 0) {
                    // exclusive scan of the class counts, kDistClasses / 32 per lane
                    int cnt[kDistClasses / 32], sum = 0;
#pragma unroll
                    for (int q = 0; q < kDistClasses / 32; ++q) {
                        cnt[q] = walk.hist[lane * (kDistClasses / 32) + q];
                        sum += cnt[q];
                    }
                    int incl = sum;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int t = __shfl_up_sync(kFull, incl, off);
                        if (lane >= off)
                            incl += t;
                    }
                    int run = incl - sum;
#pragma unroll
                    for (int q = 0; q < kDistClasses / 32; ++q) {
                        walk.hist[lane * (kDistClasses / 32) + q] = run;
                        run += cnt[q];
                    }
                }
                __syncthreads();
                for (int i = tid; i < n_smem; i += kThreads) {
                    const int cr = cls_rank[i];
                    placed[walk.hist[cr >> 24] + (cr & 0xffffff)] = s_ids[i];
                }
                __syncthreads();
                for (int i = tid; i < n_smem; i += kThreads)
                    s_ids[i] = placed[i];
            }
            __syncthreads();
        }
        for (int i = tid; i < n_smem; i += kThreads) {
            const float4 *src = gbox + 2 * s_ids[i];
            cp_async16(&s_box[2 * i], src);
            cp_async16(&s_box[2 * i + 1], src + 1);
        }
        cp_async_wait_all();
        __syncthreads();

        // One-box checks over a grid of nodes.  For a fixed patch, the viewpoints
        // whose segment to it meets a convex box form a convex set (the box's
        // shadow seen from the patch), so a box that certainly blocks the
        // extreme patches from four viewpoints blocks them from their whole
        // rectangle; the one-box argument over the target plane then covers
        // every patch.  Up to 4 x 4 viewpoints of the tile are tested (the
        // nodes), one per warp with 32 boxes over the lanes, nearest first; a
        // rectangle between four nodes is decided when one box blocks all
        // four.  A tile of 256 viewpoints then takes 16 node tests where it
        // took 64 (four viewpoints x 8 boxes each), with 32 to kNodeBoxes boxes
        // instead of 8.  Viewpoints of a rectangle none of whose nodes any box
        // blocks go to the sweep at once; the others are checked one by one.
        // Measured against 64 tests per tile (and, for many patches, a
        // whole-tile test over 128 boxes): 100,000 boxes, 64 x 32 patches 4.25
        // -> 3.46 ms, 64 uneven requests 7.95 -> 7.16 ms, strict 5,000 boxes 91
        // -> 79 us; 32 boxes per node 1-5 % slower, 128 no faster.
        bool tile_blocked = pre_blocked;
        corner_tests += pre_tests;
        const int kx = min(3, (tw + 2) >> 2), ky = min(3, (iy1 - iy0 + 2) >> 2);   // rectangles per side, 0 for one viewpoint
        const int sx = kx ? (tw - 1 + kx - 1) / kx : 1, sy = ky ? (iy1 - iy0 - 1 + ky - 1) / ky : 1;
        const int nnx = kx + 1, nodes = nnx * (ky + 1);
        const int rx = max(kx, 1), rects = rx * max(ky, 1);
        unsigned closed = 0u, seen = 0u;   // rectangles: decided; with a node that some box blocks
        if (!viewer && !pre_blocked) {
            for (int b = 0; b < min(n_smem, kNodeBoxes); b += 32) {
                unsigned *mask = s_node[(b >> 5) & 1];
                for (int nd = warp; nd < nodes; nd += kWarps) {
                    const int ny = nd / nnx, nx = nd - ny * nnx;
                    const float qx = R.x_coord[ix0 + min(nx * sx, tw - 1)];
                    const float qy = R.y_coord[min(iy0 + ny * sy, iy1 - 1)];
                    const float qu = R.au == 0 ? qx : (R.au == 1 ? qy : zq);
                    const float qn = R.an == 0 ? qx : (R.an == 1 ? qy : zq);
                    const float qw = R.dims == 3 ? (R.aw == 0 ? qx : (R.aw == 1 ? qy : zq)) : 0.f;
                    bool full = false;
                    if (b + lane < n_smem) {
                        full = box_blocks_all(R, s_box[2 * (b + lane)], s_box[2 * (b + lane) + 1], qu, qn, qw);
                        corner_tests += 4;
                    }
                    const unsigned m = __ballot_sync(kFull, full);
                    if (lane == 0)
                        mask[nd] = m;
                }
                __syncthreads();   // (the masks of the batch after next reuse the buffer)
                unsigned all = 0u, any = 0u;
                if (lane < rects) {
                    const int y = lane / rx, x = lane - y * rx;
                    const int x1 = min(x + 1, kx), y1 = min(y + 1, ky) * nnx, y0 = y * nnx;
                    const unsigned m00 = mask[y0 + x], m10 = mask[y0 + x1], m01 = mask[y1 + x], m11 = mask[y1 + x1];
                    all = m00 & m10 & m01 & m11;
                    any = m00 | m10 | m01 | m11;
                }
                closed |= __ballot_sync(kFull, all != 0u);
                seen |= __ballot_sync(kFull, any != 0u);
                if (TILE_CHECK && R.blk_base >= 0) {
                    // one box for every node: kept for the tiles of this position and its neighbours
                    const unsigned whole = __reduce_and_sync(kFull, lane < nodes ? mask[lane] : kFull);
                    if (whole && tid == 0)
                        work[kWorkHeader + ar.blocker_off() + R.blk_base + ty * R.tiles_x + tx] =
                            s_ids[b + __ffs(whole) - 1];
                }
                if (closed == (1u << rects) - 1u)
                    break;
            }
            tile_blocked = closed == (1u << rects) - 1u;
        }
        if (tile_blocked) {
            for (int i = tid; i < tn; i += kThreads) {
                const int ry = (int)(((float)i + 0.5f) * inv_tw);
                put_v(R, ((long long)layer * R.ny + iy0 + ry) * R.nx + ix0 + i - ry * tw, 0.f);
            }
            if (want_bits) {   // a row of the tile is one run of words
                const int row_words = tw * R.words, rem = R.P & 31;
                const float inv_words = 1.0f / (float)R.words;   // (exact as above: row_words < 2^20)
                const unsigned last = rem ? (1u << rem) - 1u : 0xffffffffu;
                for (int y = iy0; y < iy1; ++y) {
                    const long long at = (((long long)layer * R.ny + y) * R.nx + ix0) * R.words;
                    for (int i = tid; i < row_words; i += kThreads) {
                        const int k = (int)(((float)i + 0.5f) * inv_words);   // viewpoint of word i
                        put_word(R, at + i, i - k * R.words == R.words - 1 ? last : 0xffffffffu);
                    }
                }
            }
            if (tid == 0)
                shortcuts += (unsigned)tn;
        }
        if (viewer) {
            // viewer-centric: threads take cells, one segment each
            unsigned long long tests = 0;
            unsigned rechecks = 0;
            float vmax = 0.f;
            for (int vi = tid; vi < tn; vi += kThreads) {
                const int ry = (int)(((float)vi + 0.5f) * inv_tw), ix = ix0 + vi - ry * tw, iy = iy0 + ry;
                const long long vp = ((long long)layer * R.ny + iy) * R.nx + ix;
                bool blocked;
                const float v = viewer_cell(R, s_box, n_smem, tail, count, gbox, R.x_coord[ix], R.y_coord[iy],
                                            R.dims == 3 ? zq : 0.f, blocked, tests, rechecks, sc.n_boxes);
                put_v(R, vp, v);
                if (want_bits)
                    put_word(R, vp, blocked ? 1u : 0u);
                vmax = fmaxf(vmax, v);
            }
            for (int off = 16; off > 0; off >>= 1)
                tests += __shfl_xor_sync(kFull, tests, off);
            rechecks = __reduce_add_sync(kFull, rechecks);
            const unsigned vmax_bits = __reduce_max_sync(kFull, __float_as_uint(vmax));   // v >= 0
            if (lane == 0) {
                atomicMax(&R.stats->vmax_bits, vmax_bits);
                if (tests)
                    atomicAdd(&R.stats->slab_tests, tests);
                if (rechecks)
                    atomicAdd(&R.stats->rechecked, (unsigned long long)rechecks);
            }
        }
        // the viewpoints: decided, behind the target, open, or to check
        if (!viewer && !tile_blocked) {
            const float inv_sx = 1.0f / (float)sx, inv_sy = 1.0f / (float)sy;
            for (int base = 0; base < tn; base += kThreads) {
                const int vi = base + tid;
                bool open = false, check = false, hide = false;
                int xy = 0;
                if (vi < tn) {
                    const int y = (int)(((float)vi + 0.5f) * inv_tw), x = vi - y * tw;
                    xy = x | (y << 8);
                    // the rectangles that hold it: two along a side for a viewpoint on an inner node line
                    const int xa = min((int)(((float)x + 0.5f) * inv_sx), rx - 1);
                    const int ya = min((int)(((float)y + 0.5f) * inv_sy), max(ky, 1) - 1);
                    unsigned in = 1u << (ya * rx + xa);
                    if (xa > 0 && x == xa * sx)
                        in |= in >> 1;
                    if (ya > 0 && y == ya * sy)
                        in |= in >> rx;
                    const int ix = ix0 + x, iy = iy0 + y;
                    if (closed & in) {
                        hide = true;
                        ++shortcuts;
                    } else if (want_bits || facing(R, R.an == 0 ? R.x_coord[ix] : (R.an == 1 ? R.y_coord[iy] : zq))) {
                        check = (seen & in) != 0u;
                        open = !check;
                    }
                    if (!open && !check)
                        put_v(R, ((long long)layer * R.ny + iy) * R.nx + ix, 0.f);
                }
                const unsigned mo = __ballot_sync(kFull, open), mc = __ballot_sync(kFull, check);
                int at_o = 0, at_c = 0;
                if (lane == 0 && mo)
                    at_o = atomicAdd(&sm.n_und, __popc(mo));
                if (lane == 0 && mc)
                    at_c = atomicAdd(&s_next, __popc(mc));
                at_o = __shfl_sync(kFull, at_o, 0);
                at_c = __shfl_sync(kFull, at_c, 0);
                const unsigned below = (1u << lane) - 1u;
                if (open && IN_BOUNDS(at_o + __popc(mo & below), kMaxTileViewpoints, R.stats))
                    s_und[at_o + __popc(mo & below)] = (unsigned short)xy;
                if (check && IN_BOUNDS(at_c + __popc(mc & below), kMaxTileViewpoints, R.stats))
                    s_scratch.check[at_c + __popc(mc & below)] = (unsigned short)xy;
                if (want_bits) {   // the decided ones' words, a viewpoint at a time
                    unsigned mh = __ballot_sync(kFull, hide);
                    while (mh) {
                        const int at = __shfl_sync(kFull, xy, __ffs(mh) - 1);
                        mh &= mh - 1;
                        const long long vp = ((long long)layer * R.ny + iy0 + (at >> 8)) * R.nx + ix0 + (at & 255);
                        for (int wd = lane; wd < R.words; wd += 32) {
                            const int rem = R.P - 32 * wd;
                            put_word(R, vp * R.words + wd, rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u));
                        }
                    }
                }
            }
            __syncthreads();
            // checked one by one, four per warp: lanes as 4 viewpoints x the 8 nearest boxes
            const int n_check = s_next, sub = lane >> 3, bl = lane & 7, nb8 = min(n_smem, 8);
            for (int k0 = 4 * warp; k0 < n_check; k0 += 4 * kWarps) {
                const int k = k0 + sub;
                bool full = false;
                long long vp = 0;
                int xy = 0;
                if (k < n_check) {
                    xy = s_scratch.check[k];
                    const int ix = ix0 + (xy & 255), iy = iy0 + (xy >> 8);
                    vp = ((long long)layer * R.ny + iy) * R.nx + ix;
                    const float qx = R.x_coord[ix], qy = R.y_coord[iy];
                    const float qu = R.au == 0 ? qx : (R.au == 1 ? qy : zq);
                    const float qn = R.an == 0 ? qx : (R.an == 1 ? qy : zq);
                    const float qw = R.dims == 3 ? (R.aw == 0 ? qx : (R.aw == 1 ? qy : zq)) : 0.f;
                    if (bl < nb8) {
                        full = box_blocks_all(R, s_box[2 * bl], s_box[2 * bl + 1], qu, qn, qw);
                        corner_tests += 4;
                    }
                }
                const unsigned m = __ballot_sync(kFull, full);
                if (k >= n_check)
                    continue;
                if ((m >> (8 * sub)) & 0xffu) {
                    if (bl == 0) {
                        put_v(R, vp, 0.f);
                        ++shortcuts;
                    }
                    if (want_bits)
                        for (int wd = bl; wd < R.words; wd += 8) {
                            const int rem = R.P - 32 * wd;
                            put_word(R, vp * R.words + wd, rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u));
                        }
                } else if (bl == 0) {
                    const int at = atomicAdd(&sm.n_und, 1);
                    if (IN_BOUNDS(at, kMaxTileViewpoints, R.stats))
                        s_und[at] = (unsigned short)xy;
                }
            }
        }
        __syncthreads();
        int n_und = (viewer || tile_blocked) ? 0 : sm.n_und;
        // Work sharing (share == 1): the tile's open viewpoints go to the
        // second pass in chunks, with the tile's candidate list: swept here,
        // a few hundred tiles of mostly visible viewpoints set the end of the
        // launch (100-290 us each against 17 us for the median tile).  What
        // would pass a cap of the arena stays, as do lists so long that the pool's
        // counter could pass 2^31 with one from every resident block.
        if (share == 1 && spill_slot >= 0 && n_und > 0 && count <= kPublishMax) {
            int *arena = work + kWorkHeader;
            if (tid == 0) {
                const int want = (n_und + kChunkVp - 1) / kChunkVp;
                int rec = ar.rec_cap, base = 0, got = 0, off = 0;
                // counters move only while their caps are not reached, and all at
                // once (one round trip, not three): a tile whose record or ids did
                // not fit leaves its chunks empty
                int *ctr = work + 4 * round;
                if (__ldcg(ctr + 1) < ar.rec_cap && __ldcg(ctr + 4) < ar.pool_ints &&
                    __ldcg(ctr + 2) < ar.chunk_cap) {
                    rec = atomicAdd(ctr + 1, 1);
                    off = atomicAdd(ctr + 4, count);
                    base = atomicAdd(ctr + 2, want);
                    got = max(0, min(want, ar.chunk_cap - base));
                    if (rec >= ar.rec_cap || off > ar.pool_ints - count) {
                        for (int i = 0; i < got; ++i)
                            if (IN_BOUNDS(base + i, ar.chunk_cap, R.stats))
                                arena[(size_t)kChunkInts * (base + i)] = 0;
                        got = 0;
                    }
                    if (got > 0 && !CHECKED(publication_in_bounds(ar, rec, base, got, off, count), R.stats))
                        got = 0;
                }
                sm.pub[0] = rec;
                sm.pub[1] = base;
                sm.pub[2] = got;
                sm.pub[3] = off;
                s_next2 = min(n_und, got * kChunkVp);   // the tile keeps the rest
                s_full = stop_at < INT_MAX &&
                         (got < want || base + want > stop_at || off > ar.pool_ints - (ar.pool_ints >> 3));
                s_shared += (unsigned)s_next2;
            }
            __syncthreads();
            const int pub_n = sm.pub[2];
            if (pub_n > 0) {
                const int rec = sm.pub[0], pub_base = sm.pub[1], off = sm.pub[3];
                int *rp = arena + ar.rec_off() + (size_t)kRecInts * rec;
                int *ids = arena + ar.pool_off() + off;
                if (tid == 0) {
                    rp[0] = s_req_idx;
                    rp[1] = count;
                    rp[2] = off;
                    rp[3] = layer;
                    rp[4] = ix0;
                    rp[5] = iy0;
                }
                for (int i = tid; i < count; i += kThreads) {
                    const int id = i < n_smem ? s_ids[i] : tail[i - n_smem];
                    ids[i] = IN_BOUNDS(id, sc.n_boxes, R.stats) ? id : 0;
                }
                for (int i = tid; i < pub_n * kChunkInts; i += kThreads) {
                    const int j = i / kChunkInts, r = i - j * kChunkInts, k = j * kChunkVp + 2 * (r - 1);
                    const int n_j = min(kChunkVp, n_und - j * kChunkVp);
                    const unsigned a = s_und[min(max(k, 0), kMaxTileViewpoints - 1)];
                    const unsigned b = s_und[min(max(k + 1, 0), kMaxTileViewpoints - 1)];
                    arena[(size_t)kChunkInts * (pub_base + j) + r] =
                        r == 0 ? rec * 32 + n_j : (int)(a | (b << 16));
                }
            }
        }
        if (s_next2 < n_und)
            sweep_kept(R, s_scratch, s_box, n_smem, tail, count, gbox, s_und, &s_next2, n_und, ix0, iy0, layer,
                       sc.n_boxes);
        if (tid == 0) {
            s_listed += (unsigned)count;
            sm.item = -2;   // one_tile: the next round exits
        }
        __syncthreads();
    }
    flush();
    if (one_tile && tid == 0 && spill_slot >= 0)
        atomicExch(&spill_busy[spill_slot], 0);
}

// The second pass: the chunks that the tile pass published, by warps of their
// own.  A chunk was a block's work before (its list staged by the block, its
// warps waiting at its end for the slowest viewpoint); a warp now takes a part
// of a chunk, stages up to kWarpBoxes of the list for itself and meets no
// block barrier, so parts are as small as the launch needs: 16 viewpoints when
// there are many chunks, down to 1 when there are fewer than kPartsPerWarp
// parts per warp (2: 4 or 6 parts were 8 % slower on a strict map, 1 was 4 to 8 %
// slower on maps with bits).  What a warp knows of its part lies in shared memory and is
// read where it is used: the sweep needs the registers (in registers it
// spilled 200 bytes and issued 10 % more instructions).
//
// Bound by instruction issue (79 % of the slots; 60 % with 5,000 boxes, where
// the loads that begin a part show).  Against chunks by blocks (both passes): 96
// x 83 x 3 viewpoints, two-sided, 45 x 13 patches 92 -> 60 us; 64 x 64, 8 x 4
// patches 44 -> 36 us; 2D 128 x 128 48 -> 41 us; 64 uneven requests 8.92 -> 8.71
// ms.  Since then the part's viewpoints are set up one per lane, rows are staged
// once per layer and the measure takes two rows per operation: 64 requests 7.19
// -> 6.16 ms, 100,000 boxes, 64 x 32 patches 3.44 -> 3.14 ms.  6 blocks per SM (80
// registers): 7 spill (+6 %), 5 leave latency open (+8 %).
template <bool EXTRA>
__global__ void __launch_bounds__(kThreads, kSweepBlocks)
k_sweep(DevScene sc, const DevRequest *__restrict__ reqs, int n_req, int *__restrict__ work, Arena ar, int round)
{
    after_previous_kernel();
    struct Mine {   // one warp's: a single base address, the rest are constant offsets
        WarpScratch scratch;
        float4 boxes[2 * kWarpBoxes];
        DevRequest req;
        float4 q[kChunkVp];   // the part's viewpoints in the target frame; w: 1 in front of the target
        long long vp[kChunkVp];
        int list[8];   // the record: request, count, offset of the ids, layer, tile origin
    };
    __shared__ __align__(16) Mine s_mine[kWarps];
    const int lane = threadIdx.x & 31;
    Mine &mine = s_mine[threadIdx.x >> 5];
    WarpScratch &W = mine.scratch;
    DevRequest &R = mine.req;
    float4 *boxes = mine.boxes;
    const int *arena = work + kWorkHeader;
    int *ctr = work + 4 * round;
    const int n_chunks = min(ctr[2], ar.chunk_cap);
    if (n_chunks == 0)
        return;
    const int warps = (int)gridDim.x * kWarps;
    int part_log = 0;   // parts per chunk
    while (part_log < 4 && (n_chunks << part_log) < kPartsPerWarp * warps)
        ++part_log;
    const int part_vp = kChunkVp >> part_log;
    const volatile int *list = mine.list;   // read where it is used: registers are scarce in the sweep
    int cur_rec = -1;
    if (lane == 0)
        mine.list[0] = -1;
    __syncwarp();
    LaneMap M{};
    for (;;) {
        int item = 0;
        if (lane == 0)
            item = atomicAdd(ctr + 3, 1);
        item = __shfl_sync(kFull, item, 0);
        if ((item >> part_log) >= n_chunks)
            break;
        const int *chunk = arena + (size_t)kChunkInts * (item >> part_log);
        if (!IN_BOUNDS(item >> part_log, ar.chunk_cap, reqs[0].stats) ||
            !CHECKED(chunk_in_bounds(ar, chunk[0]), reqs[0].stats))
            continue;
        const int rec = chunk[0] >> 5;
        const int first = (item & ((1 << part_log) - 1)) * part_vp, n = min((chunk[0] & 31) - first, part_vp);
        if (n <= 0)
            continue;
        __syncwarp();   // the viewpoints before are done with the item's shared memory
        const int at = lane < n ? reinterpret_cast<const unsigned short *>(chunk + 1)[first + lane] : 0;
        if (rec != cur_rec) {
            if (!CHECKED(record_in_bounds(ar, arena + ar.rec_off() + (size_t)kRecInts * rec, reqs, n_req, sc.n_boxes),
                         reqs[0].stats))
                continue;
            cur_rec = rec;
            const int old_req = list[0];
            __syncwarp();
            if (lane < 8)
                mine.list[lane] = arena[ar.rec_off() + (size_t)kRecInts * rec + lane];
            __syncwarp();
            if (list[0] != old_req) {
                const int *src = reinterpret_cast<const int *>(reqs + list[0]);
                for (int i = lane; i < (int)(sizeof(DevRequest) / sizeof(int)); i += 32)
                    reinterpret_cast<int *>(&R)[i] = src[i];
                if (lane == 0)
                    W.rw_of = __int_as_float(0x7fffffff);
                __syncwarp();
                M = lane_map(R);
            }
            const float4 *gbox = sc.boxes[R.perm];
            for (int i = lane; i < min(list[1], kWarpBoxes); i += 32) {
                const int id = arena[ar.pool_off() + list[2] + i];
                if (!IN_BOUNDS(id, sc.n_boxes, R.stats)) {   // an empty box
                    boxes[2 * i] = make_float4(f_inf(), f_inf(), f_inf(), 0.f);
                    boxes[2 * i + 1] = make_float4(-f_inf(), -f_inf(), -f_inf(), 0.f);
                    continue;
                }
                boxes[2 * i] = __ldg(&gbox[2 * id]);
                boxes[2 * i + 1] = __ldg(&gbox[2 * id + 1]);
            }
        }
        if (lane < n) {   // one per lane: 45 instructions for all of them
            int ix = list[4] + (at & 255), iy = list[5] + (at >> 8);
            if (!CHECKED(viewpoint_in_bounds(R, ix, iy), R.stats))
                ix = iy = 0;
            const float3 q = in_target_frame(R, R.x_coord[ix], R.y_coord[iy], R.z_coord[list[3]]);
            mine.q[lane] = make_float4(q.x, q.y, q.z, facing(R, q.y) ? 1.f : 0.f);
            mine.vp[lane] = ((long long)list[3] * R.ny + iy) * R.nx + ix;
        }
        __syncwarp();
        unsigned tests = 0, corners = 0, rechecks = 0, shortcuts = 0;
        float vmax = 0.f;
        for (int k = 0; k < n; ++k) {
            const float4 q = mine.q[k];
            const float v = sweep_one<EXTRA>(R, M, make_float3(q.x, q.y, q.z), q.w != 0.f, mine.vp[k], boxes, kWarpBoxes,
                                             Tail{arena + ar.pool_off() + list[2] + kWarpBoxes, 4}, list[1],
                                             sc.boxes[R.perm], W, tests, corners, rechecks, shortcuts, sc.n_boxes);
            vmax = fmaxf(vmax, v);
        }
        rechecks = __reduce_add_sync(kFull, rechecks);
        // the lanes' tests, in two halves that cannot overflow
        const unsigned low = __reduce_add_sync(kFull, tests & 0xffffu), high = __reduce_add_sync(kFull, tests >> 16);
        if (lane == 0) {
            if (vmax > 0.f)
                atomicMax(&R.stats->vmax_bits, __float_as_uint(vmax));
            if (low | high)
                atomicAdd(&R.stats->slab_tests, ((unsigned long long)high << 16) + low);
            if (corners)
                atomicAdd(&R.stats->corner_tests, (unsigned long long)corners);
            if (shortcuts)
                atomicAdd(&R.stats->shortcut_viewpoints, (unsigned long long)shortcuts);
            if (rechecks)
                atomicAdd(&R.stats->rechecked, (unsigned long long)rechecks);
        }
    }
}

// Launch prologue: the work counters, every request's counters, and -1 in the
// launch's part of the blocker table.
__device__ __forceinline__ void prologue(const DevRequest *reqs, int n_req, int *__restrict__ work,
                                         int *__restrict__ blockers, int n_blockers)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    if (t < kWorkHeader)
        work[t] = 0;
    constexpr int kStatWords = (int)(sizeof(vcm_stats) / sizeof(unsigned));
    for (int i = t; i < n_req * kStatWords; i += nt)
        reinterpret_cast<unsigned *>(reqs[i / kStatWords].stats)[i % kStatWords] = 0u;
    for (int i = t; i < n_blockers; i += nt)
        blockers[i] = -1;
}
__global__ void k_prologue(const DevRequest *__restrict__ reqs, int n_req, int *__restrict__ work,
                           int *__restrict__ blockers, int n_blockers)
{
    after_previous_kernel();
    prologue(reqs, n_req, work, blockers, n_blockers);
}

// The same for descriptors that fit a kernel's parameters: it also writes them
// to device memory.  An upload from pinned memory is a copy-engine operation
// that the first kernel waits for, and its buffer has to be waited for before
// the next call: 49 -> 36 us per 2D map of 128 x 128.
template <int BYTES>
struct DescBlob {
    uint4 v[BYTES / 16];
};
template <int BYTES>
__global__ void k_prologue_desc(const __grid_constant__ DescBlob<BYTES> blob, int n16, uint4 *__restrict__ dst, int n_req,
                                int *__restrict__ work, int *__restrict__ blockers, int n_blockers)
{
    after_previous_kernel();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += gridDim.x * blockDim.x)
        dst[i] = blob.v[i];
    prologue(reinterpret_cast<const DevRequest *>(blob.v), n_req, work, blockers, n_blockers);
}

// ---------------------------------------------------------------------------
// recoloring from stored occlusion bits (incremental gaze change)
// ---------------------------------------------------------------------------

// Values of one target-centric request from occlusion bits made earlier
// (R.bits_out is read, not written): no occlusion test, only the sides, the
// field-of-view cone, strictness and the measure.  Two passes, because the
// viewpoints that need a measure cluster in the grid:
//  1. a warp per 32 viewpoints: the side test of each and their bit words (fully
//     blocked, or in strict mode any patch blocked, gives v = 0); the others are
//     appended to a list;
//  2. one warp per listed viewpoint, lanes over patches, the warp holding
//     the bit words in registers.  The summation follows the tile kernel's:
//     a compensated sum per lane, then a fixed-order butterfly.

struct GridPoint {
    int ix, iy, layer;
};
__device__ __forceinline__ GridPoint grid_point(const DevRequest &R, unsigned vp)
{
    const unsigned nxy = (unsigned)R.nx * (unsigned)R.ny;   // the request has less than 2^31 viewpoints
    const unsigned layer = vp / nxy, rem = vp - layer * nxy, iy = rem / (unsigned)R.nx;
    return GridPoint{(int)(rem - iy * (unsigned)R.nx), (int)iy, (int)layer};
}
__device__ __forceinline__ float3 recolor_point(const DevRequest &R, const GridPoint &g)
{
    return in_target_frame(R, R.x_coord[g.ix], R.y_coord[g.iy], R.dims == 3 ? R.z_coord[g.layer] : 0.f);
}

// Pass 1 is bound by reading the bits.  A warp takes 32 viewpoints, whose words
// are one run: where a viewpoint's words are 4, 8, ... 128 and aligned, lanes read
// 16 bytes each in order and ballots say which viewpoints are all or partly
// blocked; runs of viewpoints behind the target are not read.  512^2 x 5
// viewpoints of 16 words: 24 us (27 with one viewpoint per thread, 4 bytes a time).
__global__ void __launch_bounds__(256) k_recolor_scan(const DevRequest *__restrict__ reqs, int *__restrict__ list,
                                                      int *__restrict__ n_list)
{
    after_previous_kernel();
    __shared__ DevRequest s_r;
    if (threadIdx.x == 0)
        s_r = reqs[0];
    __syncthreads();
    const DevRequest &R = s_r;
    const int lane = threadIdx.x & 31;
    const long long n = (long long)R.nx * R.ny * R.nl;
    const bool strict = (R.flags & VCM_STRICT) != 0;
    const unsigned last_mask = (R.P & 31) ? ((1u << (R.P & 31)) - 1u) : 0xffffffffu;
    const int per = R.words >> 2;   // lanes per viewpoint
    const bool wide = (R.words & 3) == 0 && per <= 32 && (per & (per - 1)) == 0 &&
                      (reinterpret_cast<uintptr_t>(R.bits_out) & 15u) == 0;
    const int per_log = wide ? __ffs(per) - 1 : 0;
    // a run of 32s of viewpoints per warp, walked along the grid's rows: the
    // divisions are for the first
    const int warps = gridDim.x * (blockDim.x >> 5), warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long groups = (n + 31) >> 5, from = groups * warp / warps, to = groups * (warp + 1) / warps;
    GridPoint g = grid_point(R, (unsigned)min(32 * from + lane, n - 1));
    for (long long base = 32 * from; base < 32 * to; base += 32) {
        const long long vp = base + lane;
        bool front = false;
        if (vp < n) {
            front = facing(R, recolor_point(R, g).y);
            g.ix += 32;
            while (g.ix >= R.nx) {
                g.ix -= R.nx;
                if (++g.iy == R.ny) {
                    g.iy = 0;
                    if (++g.layer == R.nl)   // past the last viewpoint
                        g.layer = 0;
                }
            }
        }
        const unsigned in_front = __ballot_sync(kFull, front);
        bool all_blocked = true, any_blocked = false;
        if (wide) {
            const int at_once = 32 >> per_log;   // viewpoints per load
            const unsigned run = per == 32 ? kFull : (1u << per) - 1u, some = at_once == 32 ? kFull : (1u << at_once) - 1u;
            for (int t0 = 0; t0 < per; t0 += 4) {
                // up to four loads in flight
                uint4 w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int t = t0 + q;
                    w[q] = make_uint4(0u, 0u, 0u, 0u);
                    if (t < per && ((in_front >> (t * at_once)) & some) != 0u && base + t * at_once + (lane >> per_log) < n)
                        w[q] = __ldg(reinterpret_cast<const uint4 *>(R.bits_out + base * R.words) + t * 32 + lane);
                }
                const unsigned end = (lane & (per - 1)) == per - 1 ? last_mask : 0xffffffffu;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned full =
                        __ballot_sync(kFull, (w[q].x & w[q].y & w[q].z) == 0xffffffffu && (w[q].w & end) == end);
                    const unsigned any = __ballot_sync(kFull, (w[q].x | w[q].y | w[q].z | (w[q].w & end)) != 0u);
                    if (lane / at_once == t0 + q) {   // this lane's viewpoint was among them
                        const int sh = (lane & (at_once - 1)) << per_log;
                        all_blocked = ((full >> sh) & run) == run;
                        any_blocked = ((any >> sh) & run) != 0u;
                    }
                }
            }
        } else if (front) {
            const uint32_t *words = R.bits_out + vp * R.words;
            for (int wd = 0; wd < R.words; ++wd) {
                const unsigned full = wd == R.words - 1 ? last_mask : 0xffffffffu;
                const unsigned w = __ldg(&words[wd]) & full;
                all_blocked &= w == full;
                any_blocked |= w != 0u;
            }
        }
        const bool live = front && !all_blocked && !(strict && any_blocked);
        if (vp < n && !live)
            put_v(R, vp, 0.f);
        const unsigned m = __ballot_sync(kFull, live);
        int at = 0;
        if (lane == 0 && m)
            at = atomicAdd(n_list, __popc(m));
        at = __shfl_sync(kFull, at, 0);
        if (live && IN_BOUNDS(at + __popc(m & ((1u << lane) - 1u)), n, R.stats))
            list[at + __popc(m & ((1u << lane) - 1u))] = (int)vp;
    }
}

// Pass 2 is bound by instruction issue: per open patch a term and its
// compensated sum.  Words without an open patch are skipped, the cone is
// decided for the whole target where it can be (cone_class), rows come from
// shared memory (however many there are: with 256 of them held and the others
// loaded, 7 x 300 patches took 0.76 ms for 139,000 viewpoints, now 0.62) and a lane's
// column stays put where 32 is a multiple of the columns; then a word takes 20
// operations without a branch.  512^2 x 5 viewpoints, 32 x 16 patches, 120 degree
// cone: 107 -> 54 us.
__global__ void __launch_bounds__(256) k_recolor_measure(const DevRequest *__restrict__ reqs,
                                                         const int *__restrict__ list, const int *__restrict__ n_list,
                                                         int n_rows)
{
    after_previous_kernel();
    __shared__ DevRequest s_r;
    extern __shared__ float s_w[];   // the request's rows
    if (threadIdx.x == 0)
        s_r = reqs[0];
    __syncthreads();
    const DevRequest &R = s_r;
    for (int i = threadIdx.x; i < n_rows; i += blockDim.x)
        s_w[i] = R.w_coord[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int n = *n_list;
    const int warps = gridDim.x * (blockDim.x >> 5);
    const int nu = R.nu, du = 32 % nu, dw = 32 / nu;
    const int iu0 = lane % nu, iw0 = lane / nu;
    const unsigned last_mask = (R.P & 31) ? ((1u << (R.P & 31)) - 1u) : 0xffffffffu;
    const int n_words = R.words;
    const bool is3d = R.dims == 3;
    float vmax = 0.f;
    for (int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        const int vq = list[i];
        const float3 p = recolor_point(R, grid_point(R, (unsigned)vq));
        const float qu = p.x, qn = p.y, qw = p.z;
        const uint32_t *words = R.bits_out + (long long)vq * n_words;
        const float rn = qn - R.p_n;
        const float m_s = R.measure * ((R.flags & VCM_TWO_SIDED) ? fabsf(rn) : R.sn * rn);
        const int cone = R.cone ? cone_class(R, qu, qn, qw) : kConeIn;
        float sum = 0.f, comp = 0.f;
        // a term joins by a two-sum of the larger and the smaller (both are >= 0)
        auto add = [&](float term) {
            const float tsum = __fadd_rn(sum, term);
            comp += (fmaxf(sum, term) - tsum) + fminf(sum, term);
            sum = tsum;
        };
        auto word = [&](int k, unsigned &held) {   // word k's open patches; words 32 at a time, one per lane
            if ((k & 31) == 0) {
                const int wd = k + lane;
                held = wd < n_words ? ~__ldg(&words[wd]) & (wd == n_words - 1 ? last_mask : 0xffffffffu) : 0u;
            }
            return __shfl_sync(kFull, held, k & 31);
        };
        unsigned held = 0u;
        float ru = qu - __ldg(&R.u_coord[iu0]), col_d2 = fmaf(ru, ru, rn * rn);
        if (cone == kConeIn && is3d && du == 0) {
            // the lane's column stays; a closed patch adds +0, which changes nothing
            for (int k = 0; k < n_words; ++k) {
                const unsigned open = word(k, held);
                if (open) {
                    const float rw = qw - s_w[min(iw0 + k * dw, R.nw - 1)];
                    const float ir = rsqrt_normal(fmaf(rw, rw, col_d2));
                    const float term = m_s * (ir * ir * ir);
                    add((open >> lane) & 1u ? term : 0.f);
                }
            }
        } else if (cone != kConeOut) {
            int iu = iu0, iw = iw0;
            for (int k = 0; k < n_words; ++k) {
                const unsigned open = word(k, held);
                if (du) {   // (otherwise the lane's column stays)
                    ru = qu - __ldg(&R.u_coord[iu]);
                    col_d2 = fmaf(ru, ru, rn * rn);
                }
                if (open) {
                    if ((open >> lane) & 1u) {
                        const float rw = qw - s_w[iw];
                        if (cone == kConeIn || in_cone_inline(R, ru, rn, rw)) {
                            const float d2 = fmaf(rw, rw, col_d2);
                            const float ir = rsqrt_normal(d2);
                            add(is3d ? m_s * (ir * ir * ir) : m_s / d2);
                        }
                    }
                }
                // the lane's next patch: 32 further in row-major order
                iu += du;
                iw += dw;
                if (iu >= nu) {
                    iu -= nu;
                    ++iw;
                }
            }
        }
        float v = sum + comp;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            v += __shfl_xor_sync(kFull, v, off);
        if (lane == 0)
            put_v(R, vq, v);
        vmax = fmaxf(vmax, v);
    }
    if (lane == 0 && vmax > 0.f)
        atomicMax(&R.stats->vmax_bits, __float_as_uint(vmax));
}

// ---------------------------------------------------------------------------
// colors
// ---------------------------------------------------------------------------

// Color of one value (Def. 1 normalisation): level 0 for v = 0, else
// 1 + floor((L - 1) v / v_ref) capped at L - 1; `edge` marks a value within
// 1e-5 of an interior bin edge.
__device__ __forceinline__ unsigned char quantise_one(float v, float vref, int L, bool &edge)
{
    unsigned char c = 0;
    edge = false;
    if (v > 0.f && vref > 0.f) {
        const float x = (float)(L - 1) * v / vref;
        const int f = (int)floorf(x);
        c = (unsigned char)(1 + min(L - 2, f));
        const float r = rintf(x);
        edge = r >= 1.f && r <= (float)(L - 2) && fabsf(x - r) <= 1e-5f * x;
    }
    return c;
}

// Four consecutive viewpoints per thread: one 16-byte load of values and one
// 4-byte store of colors when the four belong to one request and both
// addresses are aligned, else one at a time.  A block takes a run of
// viewpoints and looks its request up once; for each group of four on its own
// the search took more than the colors (64 requests, 46 M viewpoints: 124 -> 121
// us).
__global__ void k_quantise(const DevRequest *__restrict__ reqs, const long long *__restrict__ vp_prefix,
                           int n_req, long long total)
{
    after_previous_kernel();
    const long long groups = (total + 3) / 4;
    const long long from = groups * blockIdx.x / gridDim.x, to = groups * (blockIdx.x + 1) / gridDim.x;
    int lo_r = 0, hi_r = n_req - 1;
    while (lo_r < hi_r) {
        const int mid = (lo_r + hi_r + 1) >> 1;
        if (vp_prefix[mid] <= 4 * from)
            lo_r = mid;
        else
            hi_r = mid - 1;
    }
    int held = -1, L = 2;
    long long first = 0, n_vp = 0;
    float vref = 0.f;
    const float *v_out = nullptr;
    unsigned char *color_out = nullptr;
    vcm_stats *stats = nullptr;
    for (long long g = from + threadIdx.x; g < to; g += blockDim.x) {
        const long long i0 = 4 * g;
        while (lo_r + 1 < n_req && vp_prefix[lo_r + 1] <= i0)
            ++lo_r;
        if (lo_r != held) {
            held = lo_r;
            const DevRequest &R = reqs[lo_r];
            first = vp_prefix[lo_r];
            n_vp = vp_prefix[lo_r + 1] - first;
            stats = R.stats;
            vref = R.v_ref_given > 0.f ? R.v_ref_given : __uint_as_float(stats->vmax_bits);
            L = R.levels;
            v_out = R.v_out;
            color_out = R.color_out;
        }
        const long long local0 = i0 - first;
        if (local0 == 0)
            stats->v_ref = vref;
        const float *vsrc = v_out + local0;
        unsigned char *cdst = color_out ? color_out + local0 : nullptr;
        if (local0 + 4 <= n_vp && (reinterpret_cast<uintptr_t>(vsrc) & 15u) == 0 &&
            (reinterpret_cast<uintptr_t>(cdst) & 3u) == 0) {
            const float4 v4 = *reinterpret_cast<const float4 *>(vsrc);
            bool e0, e1, e2, e3;
            const unsigned c = (unsigned)quantise_one(v4.x, vref, L, e0) |
                               ((unsigned)quantise_one(v4.y, vref, L, e1) << 8) |
                               ((unsigned)quantise_one(v4.z, vref, L, e2) << 16) |
                               ((unsigned)quantise_one(v4.w, vref, L, e3) << 24);
            if (cdst && IN_BOUNDS(local0 + 3, n_vp, stats))
                *reinterpret_cast<unsigned *>(cdst) = c;
            const unsigned n_edge = (unsigned)e0 + (unsigned)e1 + (unsigned)e2 + (unsigned)e3;
            if (n_edge)   // rare; lanes of one warp may belong to different requests
                atomicAdd(&stats->edge_cells, n_edge);
            continue;
        }
        // one at a time: the group's last viewpoints may start the next requests
        for (long long i = i0; i < i0 + 4 && i < total; ++i) {
            while (lo_r + 1 < n_req && vp_prefix[lo_r + 1] <= i)
                ++lo_r;   // (the next group looks its request up again)
            const DevRequest &Q = reqs[lo_r];
            const long long local = i - vp_prefix[lo_r];
            const float qref = Q.v_ref_given > 0.f ? Q.v_ref_given : __uint_as_float(Q.stats->vmax_bits);
            bool edge;
            const unsigned char c = quantise_one(Q.v_out[local], qref, Q.levels, edge);
            if (Q.color_out && IN_BOUNDS(local, (long long)Q.nx * Q.ny * Q.nl, Q.stats))
                Q.color_out[local] = c;
            if (edge)
                atomicAdd(&Q.stats->edge_cells, 1u);
            if (local == 0)
                Q.stats->v_ref = qref;
        }
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------

cudaError_t init_device()
{
    static bool done[64] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev >= 0 && dev < 64 && done[dev])
        return cudaSuccess;
    const void *kernels[2] = {(const void *)k_tiles<false>, (const void *)k_tiles<true>};
    for (const void *k : kernels)
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)tiles_smem_bytes(kMaxBoxCap, kMaxBoxCap))) != cudaSuccess)
            return e;
    if (dev >= 0 && dev < 64)
        done[dev] = true;
    return cudaSuccess;
}

// Scratch for callers that cannot allocate device memory (vcm_compute_static).
// A file-scope __device__ array: every GPU that loads the library holds it
// until the process exits.  Host code must not use the symbol as a pointer;
// it asks the runtime for the array's device address once per device.
static __device__ __align__(256) unsigned char g_static_scratch[VCM_STATIC_SCRATCH_BYTES];

cudaError_t static_scratch(void **ptr, size_t *bytes)
{
    static std::mutex mu;
    static void *addr[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev < 0 || dev >= 64)
        return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> g(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        if ((e = cudaGetSymbolAddress(&p, g_static_scratch)) != cudaSuccess)
            return e;
        addr[dev] = p;
    }
    *ptr = addr[dev];
    *bytes = sizeof(g_static_scratch);
    return cudaSuccess;
}

// Launch with programmatic stream serialization (see after_previous_kernel).
// `overlap` false: an ordinary launch.
template <typename... KArgs, typename... Args>
static cudaError_t launch(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t stream, bool overlap,
                          Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

cudaError_t launch_grid_build(const float *d_lo_world, const float *d_hi_world, int n, int dims,
                              float gx0, float gy0, float cell, int gnx, int gny,
                              int *d_cell_of, int *d_count, int *d_order,
                              int *d_cell_start, float4 *const *d_perm_boxes, float4 *d_cell_lo,
                              float4 *d_cell_hi, unsigned *d_overhang_bits, cudaStream_t stream)
{
    (void)dims;
    const int n_cells = gnx * gny;
    const int tb = 256;
    cudaError_t e;
    if ((e = cudaMemsetAsync(d_count, 0, sizeof(int) * n_cells, stream)) != cudaSuccess) return e;
    if (n > 0 && (e = launch(k_box_cell, (n + tb - 1) / tb, tb, 0, stream, true, d_lo_world, d_hi_world, n, gx0, gy0,
                             1.0f / cell, gnx, gny, d_cell_of, d_count)) != cudaSuccess)
        return e;
    if (n_cells <= kScanOneMax) {
        if ((e = launch(k_scan_one, 1, kScanOneThreads, 0, stream, true, d_count, n_cells, d_cell_start,
                        d_overhang_bits)) != cudaSuccess)
            return e;
    } else {
        // its block sums live in d_cell_lo, which k_cell_bounds writes only at
        // the end (16 bytes per cell, 4 per block sum)
        const int n_scan_blocks = (n_cells + kScanChunk - 1) / kScanChunk;
        if (n_scan_blocks > 1024)
            return cudaErrorInvalidValue;
        int *block_sum = reinterpret_cast<int *>(d_cell_lo);
        if ((e = launch(k_scan_reduce, n_scan_blocks, kScanThreads, 0, stream, true, d_count, n_cells, block_sum)) !=
                cudaSuccess ||
            (e = launch(k_scan_top, 1, 1024, 0, stream, true, block_sum, n_scan_blocks, n_cells, d_cell_start,
                        d_overhang_bits)) != cudaSuccess ||
            (e = launch(k_scan_down, n_scan_blocks, kScanThreads, 0, stream, true, d_count, n_cells, block_sum,
                        d_cell_start)) != cudaSuccess)
            return e;
    }
    if (n > 0) {
        PermPtrs pp;
        for (int p = 0; p < 6; ++p)
            pp.p[p] = d_perm_boxes[p];
        if ((e = launch(k_scatter, (n + tb - 1) / tb, tb, 0, stream, true, d_cell_of, n, d_cell_start, d_count,
                        d_order)) != cudaSuccess ||
            (e = launch(k_write_boxes, (n + 127) / 128, 128, 0, stream, true, d_lo_world, d_hi_world, n, d_cell_of,
                        d_cell_start, d_order, pp)) != cudaSuccess)
            return e;
    }
    return launch(k_cell_bounds, (n_cells + tb - 1) / tb, tb, 0, stream, true, d_perm_boxes[0], d_cell_start, gnx, gny,
                  gx0, gy0, cell, d_cell_lo, d_cell_hi, d_overhang_bits);
}

// Blocks of the tile pass per SM by shared memory (the instantiations share
// their launch bounds).  The runtime's answer is kept: it is a property of the
// device and the kernel, and asking took 2 us, four times per call.
int tiles_blocks_per_sm(int box_cap, int list_cap)
{
    static std::mutex mu;
    static std::map<std::pair<int, size_t>, int> known;
    const size_t smem = tiles_smem_bytes(box_cap, std::max(list_cap, box_cap));
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return 1;
    std::lock_guard<std::mutex> g(mu);
    const auto it = known.find({dev, smem});
    if (it != known.end())
        return it->second;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_tiles<false>, kThreads, smem) != cudaSuccess)
        return 1;
    n = n > 0 ? n : 1;
    known[{dev, smem}] = n;   // (box_cap takes at most kMaxBoxCap values)
    return n;
}

int spill_id_bytes(int n_boxes) { return n_boxes < kWideIds ? 3 : 4; }

cudaError_t launch_tiles(const DevScene &sc, const DevRequest *d_reqs, const int *d_tile_prefix,
                         int n_req, int total_tiles, long long total_vp, int *d_work, int *d_spill, int grid_blocks,
                         int box_cap, bool extra, bool tile_check, int sm_count, cudaStream_t stream, bool one_tile,
                         int *d_spill_busy, bool share, int claim_rounds, const Arena &arena, int list_cap,
                         bool overlap)
{
    if (claim_rounds < 1 || claim_rounds > kClaimRounds)
        return cudaErrorInvalidValue;
    if (total_tiles <= 0)
        return cudaSuccess;
    if (box_cap < 1 || box_cap > kMaxBoxCap)
        return cudaErrorInvalidValue;
    list_cap = std::max(list_cap, box_cap);
    const size_t smem = tiles_smem_bytes(box_cap, list_cap);
    const int slots = grid_blocks;   // spill regions: the resident-block bound
    if (one_tile) {
        if (!d_spill_busy)
            return cudaErrorInvalidValue;
        grid_blocks = total_tiles;
    }
    auto kernel = tile_check ? k_tiles<true> : k_tiles<false>;
    share = share && !one_tile;
    // A launch with many more viewpoints than the arena holds runs in rounds:
    // when the arena is nearly full, each block stops after the tile it is at, the
    // second pass empties it, and the tile pass takes the queue up again.  The
    // last round runs to the queue's end whatever the arena holds; what does
    // not fit there the tiles sweep themselves, with kKeptWarps warps per block.
    // 256 requests, 49.3 M open viewpoints: 50.1 -> 35.0 ms.  A round that finds
    // nothing left costs 8 us (33.5 M viewpoints with 0.3 M open: 1.282 ms in one
    // round, 1.291 in two, 1.298 in three).  What fills an arena (12.8 M) is open
    // viewpoints, which the host does not know; launches of up to four arenas'
    // viewpoints (51 M) run in one round, for maps of cities leave 1 to 9 % open,
    // and longer ones have a round per two.  Open maps below the line pay for it,
    // though less than when the tiles kept all they could not publish and swept it
    // with every warp: 33.5 M viewpoints of 512 patches, 30 M open, 29.1 ms then,
    // 17.4 now, 13.6 in three rounds; of 2,048 patches 88.9, 48.2 and 31.4; 16.8 M
    // of 8 patches, 13.2 M open, 10.6, 7.4 and 7.1.  Static maps (an arena of
    // 0.5 M, always one round): 8.4 M viewpoints of 512 patches, all open, 12.1 ms
    // then, 7.6 now.
    const int usable = std::max(arena.chunk_cap / 2, arena.chunk_cap - grid_blocks * (kMaxTileViewpoints / kChunkVp));
    const long long rounds =
        share && total_vp > 4LL * kChunkVp * arena.chunk_cap
            ? std::min<long long>(kMaxRounds, 1 + total_vp / (2LL * kChunkVp * std::max(1, usable))) : 1;
    cudaError_t e = cudaSuccess;
    for (int r = 0; r < rounds && e == cudaSuccess; ++r) {
        e = launch(kernel, grid_blocks, kThreads, smem, stream, overlap || r > 0, sc, d_reqs, d_tile_prefix, n_req,
                   total_tiles, d_work, arena, reinterpret_cast<unsigned char *>(d_spill),
                   spill_id_bytes(sc.n_boxes), box_cap, list_cap, one_tile ? 1 : 0, d_spill_busy, slots,
                   share ? 1 : 0, claim_rounds, r + 1 < rounds ? usable : INT_MAX, r);
        if (e == cudaSuccess && share)   // the second pass, on every SM
            e = launch(extra ? k_sweep<true> : k_sweep<false>, sm_count * kSweepBlocks, kThreads, 0, stream, true,
                       sc, d_reqs, n_req, d_work, arena, r);
    }
    return e;
}

static int prologue_blocks(size_t desc_bytes, int n_req, long long n_blockers)
{
    const long long items = std::max(std::max((long long)desc_bytes / 16, 18LL * n_req), n_blockers / 8);
    return (int)std::max<long long>(1, std::min<long long>(152, (items + 255) / 256));
}

cudaError_t launch_prologue(const DevRequest *d_reqs, int n_req, int *d_work, int *d_blockers, long long n_blockers,
                            cudaStream_t stream)
{
    if (n_req <= 0)
        return cudaSuccess;
    return launch(k_prologue, prologue_blocks(0, n_req, n_blockers), 256, 0, stream, false, d_reqs, n_req, d_work,
                  d_blockers, (int)n_blockers);
}

template <int BYTES>
static cudaError_t prologue_desc(const void *h_desc, size_t bytes, void *d_desc, int n_req, int *d_work, int *d_blockers,
                                 long long n_blockers, cudaStream_t stream)
{
    DescBlob<BYTES> blob;
    std::memcpy(&blob, h_desc, bytes);
    return launch(k_prologue_desc<BYTES>, prologue_blocks(bytes, n_req, n_blockers), 256, 0, stream, true, blob,
                  (int)((bytes + 15) / 16), static_cast<uint4 *>(d_desc), n_req, d_work, d_blockers, (int)n_blockers);
}

cudaError_t launch_prologue_desc(const void *h_desc, size_t bytes, void *d_desc, int n_req, int *d_work, int *d_blockers,
                                 long long n_blockers, cudaStream_t stream)
{
    if (n_req <= 0)
        return cudaSuccess;
    if (bytes <= 4096)
        return prologue_desc<4096>(h_desc, bytes, d_desc, n_req, d_work, d_blockers, n_blockers, stream);
    if (bytes <= 16384)
        return prologue_desc<16384>(h_desc, bytes, d_desc, n_req, d_work, d_blockers, n_blockers, stream);
    if (bytes <= kDescParamBytes)
        return prologue_desc<kDescParamBytes>(h_desc, bytes, d_desc, n_req, d_work, d_blockers, n_blockers, stream);
    return cudaErrorInvalidValue;
}

cudaError_t launch_quantise(const DevRequest *d_reqs, const long long *d_vp_prefix, int n_req,
                            long long total_vp, cudaStream_t stream)
{
    if (total_vp <= 0)
        return cudaSuccess;
    long long blocks = ((total_vp + 3) / 4 + 255) / 256;   // four viewpoints per thread
    if (blocks > 152 * 16)
        blocks = 152 * 16;
    return launch(k_quantise, (int)blocks, 256, 0, stream, true, d_reqs, d_vp_prefix, n_req, total_vp);
}

cudaError_t launch_recolor(const DevRequest *d_req, long long n_vp, int n_rows, int sm_count, int *d_list, int *d_n_list,
                           cudaStream_t stream)
{
    if (n_vp <= 0)
        return cudaSuccess;
    if (n_rows < 1 || n_rows > (int)VCM_MAX_PATCHES_SIDE)
        return cudaErrorInvalidValue;
    long long blocks = (n_vp + 255) / 256;
    const long long cap = (long long)std::max(sm_count, 1) * 8;
    if (blocks > cap)
        blocks = cap;
    const cudaError_t e = launch(k_recolor_scan, (int)blocks, 256, 0, stream, true, d_req, d_list, d_n_list);
    if (e != cudaSuccess)
        return e;
    return launch(k_recolor_measure, (int)cap, 256, sizeof(float) * n_rows, stream, true, d_req, d_list, d_n_list, n_rows);
}

}  // namespace vcm
