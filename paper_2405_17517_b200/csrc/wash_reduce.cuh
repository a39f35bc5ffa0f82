// The dense comparison operators, each one pass over the stack:
//   kOpEma       PAPA's EMA, Eq. 1:  x_n <- alpha x_n + (1 - alpha) m
//   kOpAverage   the averaged model (output of Algorithm 1): out <- m
//   kOpPapaAll   PAPA-all / DART: x_n <- m
// with m = (((x_0 + x_1) + x_2) + ...)/N in binary32, each operation rounded once
// (explicit _rn intrinsics: the compiler may neither fuse nor reorder them).
//
// The unit of work is 16 bytes of every model: 4 coordinates in fp32, 8 in bf16 (tensors start on
// multiples of 8 elements, so a unit never straddles two).  [N][P] keeps a unit's N vectors in registers
// where N is small (unrolled per N), [P][N] the 4N values of a group of four coordinates (pn_in_registers says which N);
// larger populations stage them in shared memory by cp.async, sum them from there and, for the operators that write the
// stack, read them once more from there.
// Bound: HBM, except bf16 [P][N], which has two values a word to widen, round and check for NaN and is bound
// by issue slots (N = 32 249 us where the bytes take 164).  Before, a thread held four coordinates of every model (8-byte
// vectors in bf16, values of [P][N] picked out of registers), and populations not in a list of unrolled sizes went
// through local memory: EMA N = 8 bf16 ResNet-50 141 -> 133 us, [P][N] 233 -> 160; N = 7 fp32, 2^24 coordinates 671 -> 142, N = 31 [P][N],
// 2^23 coordinates 1740 -> 311; average of N = 13, fp32 ResNet-50 1029 -> 206.
#pragma once
#define WASH_SERVING_ONLY
#include "wash_shuffle_async.cuh"

namespace wash {

template <class T>
struct Unit {
    static constexpr int kElems = 16 / T::kBytes;
    static constexpr uint32_t kGroups = kElems / 4;
    // element q of a vector, widened to binary32
    static __device__ __forceinline__ float get(const uint4 &v, int q)
    {
        const uint32_t w = T::kBytes == 4 ? (q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w)
                                          : (q < 2 ? v.x : q < 4 ? v.y : q < 6 ? v.z : v.w);
        if (T::kBytes == 4) return __uint_as_float(w);
        return __uint_as_float((q & 1) ? w & 0xFFFF0000u : w << 16);
    }
    static __device__ __forceinline__ uint4 pack(const float (&r)[kElems])
    {
        if constexpr (T::kBytes == 4) return make_uint4(__float_as_uint(r[0]), __float_as_uint(r[1]), __float_as_uint(r[2]), __float_as_uint(r[3]));
        else return make_uint4(BF16::pair_from_floats(r[0], r[1]), BF16::pair_from_floats(r[2], r[3]), BF16::pair_from_floats(r[4], r[5]), BF16::pair_from_floats(r[6], r[7]));
    }
    // coordinates that exist among the unit's elements (a tensor may end inside it; the rest is padding)
    static __device__ __forceinline__ int valid(const PopView &pop, uint64_t unit, uint32_t *status)
    {
        const uint32_t g = static_cast<uint32_t>(unit) * kGroups;
        uint32_t s = __ldg(pop.tile_first + (g >> kTileShift));
        const uint32_t last = static_cast<uint32_t>(pop.n_seg) - 1u;
        while (s < last && g >= __ldg(&pop.seg[s].group_end)) ++s;
        const uint4 lo = __ldg(reinterpret_cast<const uint4 *>(pop.seg + s));   // begin, end, tensor, cgroup_begin
        if (g < lo.x || g >= lo.y) {   // table inconsistent with the row: report, touch nothing
            if (status) atomicOr(status, 1u);
            return 0;
        }
        const long long left = static_cast<long long>(__ldg(&pop.seg[s].numel)) - 4ll * (g - lo.x);
        return left >= kElems ? kElems : (left > 0 ? static_cast<int>(left) : 0);
    }
};

// One unit of the average row: m of its coordinates.
template <class T, class TOUT>
__device__ __forceinline__ void store_average(const ReduceArgs &a, uint64_t unit, int valid, const float (&m)[Unit<T>::kElems])
{
    constexpr int kElems = Unit<T>::kElems;
    const long long e0 = static_cast<long long>(unit) * kElems;
    if (valid == kElems) {
        char *out = static_cast<char *>(a.out) + e0 * TOUT::kBytes;
#pragma unroll
        for (int q = 0; q < kElems; q += 4) TOUT::store_group(out + q * TOUT::kBytes, TOUT::pack_floats(m[q], m[q + 1], m[q + 2], m[q + 3]));
    } else {
#pragma unroll
        for (int q = 0; q < kElems; ++q)
            if (q < valid) TOUT::store_elem(a.out, e0 + q, TOUT::from_float(m[q]));
    }
}

// [N][P], a thread per unit, its N vectors in registers, all loads in flight at once.
template <class T, class TOUT, int OP, int N>
__global__ void __launch_bounds__(256) regs_np_kernel(const __grid_constant__ ReduceArgs a)
{
    await_previous();
    let_next_start();
    constexpr int kElems = Unit<T>::kElems;
    const uint64_t unit = a.group_lo / Unit<T>::kGroups + static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (unit * Unit<T>::kGroups >= a.group_hi) return;
    const size_t row = static_cast<size_t>(a.pop.padded_P) * T::kBytes;
    char *out = static_cast<char *>(a.stack) + unit * 16;
    uint4 v[N];
#pragma unroll
    for (int n = 0; n < N; ++n) v[n] = F32::load_group(out + n * row);
    const int valid = Unit<T>::valid(a.pop, unit, a.status);
    if (valid == 0) return;
    float m[kElems];
#pragma unroll
    for (int q = 0; q < kElems; ++q) {
        m[q] = Unit<T>::get(v[0], q);
#pragma unroll
        for (int n = 1; n < N; ++n) m[q] = __fadd_rn(m[q], Unit<T>::get(v[n], q));
        m[q] = __fdiv_rn(m[q], static_cast<float>(N));
        if (OP == kOpEma) m[q] = __fmul_rn(a.one_minus_alpha, m[q]);
    }
    if constexpr (OP == kOpAverage) store_average<T, TOUT>(a, unit, valid, m);
    else if (valid == kElems) {
        const uint4 all = Unit<T>::pack(m);   // PAPA-all: every model's vector
#pragma unroll
        for (int n = 0; n < N; ++n, out += row) {
            if constexpr (OP == kOpPapaAll) *reinterpret_cast<uint4 *>(out) = all;
            else {
                float r[kElems];
#pragma unroll
                for (int q = 0; q < kElems; ++q) r[q] = __fadd_rn(__fmul_rn(a.alpha, Unit<T>::get(v[n], q)), m[q]);
                *reinterpret_cast<uint4 *>(out) = Unit<T>::pack(r);
            }
        }
    } else {
#pragma unroll
        for (int n = 0; n < N; ++n, out += row) {
#pragma unroll
            for (int q = 0; q < kElems; ++q)
                if (q < valid) T::store_elem(out, q, T::from_float(OP == kOpPapaAll ? m[q] : __fadd_rn(__fmul_rn(a.alpha, Unit<T>::get(v[n], q)), m[q])));
        }
    }
}

// [P][N], small N: a thread per group of four coordinates, its 4N contiguous values in registers.
template <class T, class TOUT, int OP, int N>
__global__ void __launch_bounds__(256) regs_pn_kernel(const __grid_constant__ ReduceArgs a)
{
    await_previous();
    let_next_start();
    const uint64_t g = a.group_lo + static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (g >= a.group_hi) return;
    constexpr int kVec = 4 * T::kBytes;
    char *group = group_vec_ptr<T, kLayoutPN>(a.stack, a.pop, g, 0);
    typename T::vec v[N];   // element f of the group = (coordinate f / N, model f % N)
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = T::load_group(group + j * kVec);
    const int valid = find_group(a.pop, static_cast<uint32_t>(g), a.status).valid;
    if (valid == 0) return;
    float m[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        m[c] = T::to_float(T::get(v[c * N / 4], c * N % 4));
#pragma unroll
        for (int n = 1; n < N; ++n) m[c] = __fadd_rn(m[c], T::to_float(T::get(v[(c * N + n) / 4], (c * N + n) % 4)));
        m[c] = __fdiv_rn(m[c], static_cast<float>(N));
        if (OP == kOpEma) m[c] = __fmul_rn(a.one_minus_alpha, m[c]);
    }
    const long long e0 = 4ll * static_cast<long long>(g);
    if constexpr (OP == kOpAverage) {
        if (valid == 4) TOUT::store_group(static_cast<char *>(a.out) + e0 * TOUT::kBytes, TOUT::pack_floats(m[0], m[1], m[2], m[3]));
        else {
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (c < valid) TOUT::store_elem(a.out, e0 + c, TOUT::from_float(m[c]));
        }
    } else {
        const auto updated = [&](int f) -> float {
            return OP == kOpPapaAll ? m[f / N] : __fadd_rn(__fmul_rn(a.alpha, T::to_float(T::get(v[f / 4], f % 4))), m[f / N]);
        };
        if (valid == 4) {
#pragma unroll
            for (int j = 0; j < N; ++j)
                T::store_group(group + j * kVec, T::pack_floats(updated(4 * j), updated(4 * j + 1), updated(4 * j + 2), updated(4 * j + 3)));
        } else {   // a tensor's ragged end: its padding is not written
#pragma unroll
            for (int f = 0; f < 3 * N; ++f)
                if (f < valid * N) T::store_elem(group, f, T::from_float(updated(f)));
        }
    }
}

// [N][P], any N: a thread stages the vectors of `per_thread` <= 4 units,
// blockDim.x apart, and reads nobody else's, so the kernel has no barrier.  Image: vector n of unit u at [u][n][thread].
template <class T, class TOUT, int OP>
__global__ void __launch_bounds__(64, 20) staged_np_kernel(const __grid_constant__ ReduceArgs a, int per_thread)
{
    await_previous();
    let_next_start();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int kElems = Unit<T>::kElems;
    const int n_models = a.pop.N;
    const uint32_t T_ = blockDim.x;
    const size_t row = static_cast<size_t>(a.pop.padded_P) * T::kBytes;
    const uint64_t first = a.group_lo / Unit<T>::kGroups + static_cast<uint64_t>(blockIdx.x) * T_ * per_thread + threadIdx.x;
    const uint64_t unit_hi = a.group_hi / Unit<T>::kGroups;
    char *stack = static_cast<char *>(a.stack);
    uint32_t dst = smem_addr(smem_raw) + threadIdx.x * 16;
    for (int u = 0; u < per_thread; ++u) {
        const uint64_t unit = first + static_cast<uint64_t>(u) * T_;
        if (unit >= unit_hi) break;
        const char *src = stack + unit * 16;
#pragma unroll 4
        for (int n = 0; n < n_models; ++n, src += row, dst += T_ * 16) cp_async<16>(dst, src);
    }
    uint32_t valids = 0;   // four bits per unit
    for (int u = 0; u < per_thread; ++u) {
        const uint64_t unit = first + static_cast<uint64_t>(u) * T_;
        if (unit >= unit_hi) break;
        valids |= static_cast<uint32_t>(Unit<T>::valid(a.pop, unit, a.status)) << (4 * u);
    }
    cp_async_wait_all();
    const uint4 *image = reinterpret_cast<const uint4 *>(smem_raw) + threadIdx.x;
    const float count = static_cast<float>(n_models);
    for (int u = 0; u < per_thread; ++u, image += n_models * T_) {
        const int valid = static_cast<int>((valids >> (4 * u)) & 15u);
        if (valid == 0) continue;
        const uint64_t unit = first + static_cast<uint64_t>(u) * T_;
        float m[kElems];
        {
            const uint4 v = image[0];
#pragma unroll
            for (int q = 0; q < kElems; ++q) m[q] = Unit<T>::get(v, q);
        }
#pragma unroll 4
        for (int n = 1; n < n_models; ++n) {
            const uint4 v = image[n * T_];
#pragma unroll
            for (int q = 0; q < kElems; ++q) m[q] = __fadd_rn(m[q], Unit<T>::get(v, q));
        }
#pragma unroll
        for (int q = 0; q < kElems; ++q) {
            m[q] = __fdiv_rn(m[q], count);
            if (OP == kOpEma) m[q] = __fmul_rn(a.one_minus_alpha, m[q]);
        }
        char *out = stack + unit * 16;
        if constexpr (OP == kOpAverage) store_average<T, TOUT>(a, unit, valid, m);
        else if (valid == kElems) {
            const uint4 all = Unit<T>::pack(m);   // PAPA-all: every model's vector
#pragma unroll 2
            for (int n = 0; n < n_models; ++n, out += row) {
                if constexpr (OP == kOpPapaAll) *reinterpret_cast<uint4 *>(out) = all;
                else {
                    const uint4 v = image[n * T_];
                    float r[kElems];
#pragma unroll
                    for (int q = 0; q < kElems; ++q) r[q] = __fadd_rn(__fmul_rn(a.alpha, Unit<T>::get(v, q)), m[q]);
                    *reinterpret_cast<uint4 *>(out) = Unit<T>::pack(r);
                }
            }
        } else {
            for (int n = 0; n < n_models; ++n, out += row) {
                const uint4 v = image[n * T_];
#pragma unroll
                for (int q = 0; q < kElems; ++q)
                    if (q < valid) T::store_elem(out, q, T::from_float(OP == kOpPapaAll ? m[q] : __fadd_rn(__fmul_rn(a.alpha, Unit<T>::get(v, q)), m[q])));
            }
        }
    }
}

// [P][N], all three operators.  A unit's values are N contiguous vectors, element f = (coordinate f / N, model
// f % N); a warp copies the vectors of its 32 * per_thread units in the order they lie, a lane sums and
// updates its own units' vectors where they are in shared memory (a unit takes an odd number of vectors
// there, N or N + 1, so that the lanes fall into different banks), and the warp copies them back in the
// order they lie.
// kN: the population size if it is below the number of elements in a vector (a vector may then hold
// several coordinates' ends, which only unrolled code can place cheaply), else 0.
template <class T, class TOUT, int OP, int kN>
__global__ void __launch_bounds__(64, 16) dense_pn_kernel(const __grid_constant__ ReduceArgs a, int per_thread)
{
    await_previous();
    let_next_start();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int kElems = Unit<T>::kElems;
    const uint32_t N = kN ? kN : static_cast<uint32_t>(a.pop.N), pitch = N | 1u;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint4 *image = reinterpret_cast<uint4 *>(smem_raw) + static_cast<size_t>(warp) * 32u * per_thread * pitch;
    const uint64_t unit_hi = a.group_hi / Unit<T>::kGroups;
    const uint64_t first = a.group_lo / Unit<T>::kGroups + (static_cast<uint64_t>(blockIdx.x) * (blockDim.x >> 5) + warp) * 32u * per_thread;
    if (first >= unit_hi) return;   // (no barrier below covers more than the warp)
    const uint32_t units = static_cast<uint32_t>(min(static_cast<uint64_t>(32u * per_thread), unit_hi - first));
    uint4 *stack = static_cast<uint4 *>(a.stack) + first * N;
    const uint32_t dq = 32u / N, dr = 32u - dq * N;
    // vector k is vector j = k % N of unit k / N; the pair is advanced without dividing again
    {
        uint32_t unit = lane / N, j = lane - unit * N;
        const uint32_t base = smem_addr(image);
        for (uint32_t k = lane; k < units * N; k += 32) {
            cp_async<16>(base + (unit * pitch + j) * 16u, stack + k);
            unit += dq;
            j += dr;
            if (j >= N) { j -= N; ++unit; }
        }
    }
    uint32_t valids = 0;
    for (int u = 0; u < per_thread; ++u)
        if (32u * u + lane < units) valids |= static_cast<uint32_t>(Unit<T>::valid(a.pop, first + 32u * u + lane, a.status)) << (4 * u);
    cp_async_wait_all();
    __syncwarp();
    const float count = static_cast<float>(N);
    for (int u = 0; u < per_thread; ++u) {
        const int valid = static_cast<int>((valids >> (4 * u)) & 15u);
        uint4 *mine = image + (32u * u + lane) * pitch;
        if (valid) {
            float m[kElems];   // run-time N: the finished coordinates are shifted through m
            uint32_t n = 0;
            auto finished = [&](float s) -> float {
                const float mean = __fdiv_rn(s, count);
                return OP == kOpEma ? __fmul_rn(a.one_minus_alpha, mean) : mean;
            };
            auto shift = [&]() {
#pragma unroll
                for (int i = 0; i + 1 < kElems; ++i) m[i] = m[i + 1];
            };
            if constexpr (kN != 0) {
#pragma unroll
                for (int j = 0; j < kN; ++j) {
                    const uint4 v = mine[j];
#pragma unroll
                    for (int q = 0; q < kElems; ++q) {
                        const int f = j * kElems + q, c = f / kN;
                        m[c] = f % kN == 0 ? Unit<T>::get(v, q) : __fadd_rn(m[c], Unit<T>::get(v, q));
                    }
                }
#pragma unroll
                for (int c = 0; c < kElems; ++c) m[c] = finished(m[c]);
            } else {
                float s = 0.f;
                for (uint32_t j = 0; j < N; ++j) {
                    const uint4 v = mine[j];
                    if (n + kElems <= N) {   // one coordinate's values
                        s = n == 0 ? Unit<T>::get(v, 0) : __fadd_rn(s, Unit<T>::get(v, 0));
#pragma unroll
                        for (int q = 1; q < kElems; ++q) s = __fadd_rn(s, Unit<T>::get(v, q));
                        n += kElems;
                        if (n == N) {
                            n = 0;
                            shift();
                            m[kElems - 1] = finished(s);
                        }
                    } else {                 // the end of one, the beginning of the next
                        const uint32_t rest = N - n;
#pragma unroll
                        for (int q = 0; q < kElems; ++q) {
                            if (q == static_cast<int>(rest)) {
                                shift();
                                m[kElems - 1] = finished(s);
                                s = Unit<T>::get(v, q);
                            } else s = __fadd_rn(s, Unit<T>::get(v, q));
                        }
                        n = kElems - rest;
                    }
                }
            }
            if constexpr (OP == kOpAverage) store_average<T, TOUT>(a, first + 32u * u + lane, valid, m);
            else if (valid == kElems) {
                auto updated = [&](const uint4 &v, int q, float mean) -> float {
                    return OP == kOpPapaAll ? mean : __fadd_rn(__fmul_rn(a.alpha, Unit<T>::get(v, q)), mean);
                };
                if constexpr (kN != 0) {
#pragma unroll
                    for (int j = 0; j < kN; ++j) {
                        const uint4 v = mine[j];
                        float r[kElems];
#pragma unroll
                        for (int q = 0; q < kElems; ++q) r[q] = updated(v, q, m[(j * kElems + q) / kN]);
                        mine[j] = Unit<T>::pack(r);
                    }
                } else {
                    for (uint32_t j = 0; j < N; ++j) {
                        const uint4 v = mine[j];
                        float r[kElems];
                        const uint32_t rest = N - n;   // elements of the current coordinate left; at least one
#pragma unroll
                        for (int q = 0; q < kElems; ++q) r[q] = updated(v, q, static_cast<uint32_t>(q) < rest ? m[0] : m[1]);
                        n += kElems;
                        if (n >= N) {
                            n -= N;
                            shift();
                        }
                        mine[j] = Unit<T>::pack(r);
                    }
                }
            } else {   // a tensor's ragged end: its padding is not written
                n = 0;
                for (uint32_t f = 0; f < static_cast<uint32_t>(valid) * N; ++f) {
                    const float x = T::to_float(T::load_elem(mine, f));
                    T::store_elem(stack + (static_cast<size_t>(32u * u) + lane) * N, f, T::from_float(OP == kOpPapaAll ? m[0] : __fadd_rn(__fmul_rn(a.alpha, x), m[0])));
                    if (++n == N) {
                        n = 0;
                        shift();
                    }
                }
            }
        }
        if constexpr (OP != kOpAverage) {
            const uint32_t whole = __ballot_sync(0xFFFFFFFFu, valid == kElems);
            __syncwarp();   // the units are copied by other lanes than those that updated them; a vote orders no memory accesses
            uint32_t unit = lane / N, j = lane - unit * N;
            for (uint32_t k = lane; k < 32u * N; k += 32) {
                if ((whole >> unit) & 1u) stack[static_cast<size_t>(32u * u) * N + k] = image[(32u * u + unit) * pitch + j];
                unit += dq;
                j += dr;
                if (j >= N) { j -= N; ++unit; }
            }
        }
    }
}

// Units a thread stages: small populations take several, so that enough bytes are in flight.
inline int units_per_thread(int N) { return N <= 2 ? 4 : (N <= 5 ? 2 : 1); }

template <class K>
cudaError_t launch_dense(K kernel, const ReduceArgs &args, uint64_t units, int per_thread, size_t bytes_per_unit, const LaunchShape &shape, cudaStream_t stream)
{
    int threads = shape.threads > 0 && shape.threads < 64 ? 32 : 64;
    while (threads > 32 && bytes_per_unit * per_thread * threads > 44 * 1024) threads >>= 1;   // five blocks and more on an SM
    const size_t smem = bytes_per_unit * per_thread * threads;
    KernelFit fit;
    cudaError_t err = kernel_fit(reinterpret_cast<const void *>(kernel), threads, smem, &fit);
    if (err != cudaSuccess) return err;
    if (fit.occupancy < 1) return cudaErrorLaunchOutOfResources;
    const uint64_t per_block = static_cast<uint64_t>(threads) * per_thread, grid = (units + per_block - 1) / per_block;
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    return launch_chained(kernel, static_cast<unsigned>(grid), threads, smem, stream, args, per_thread);
}

// [N][P]: the largest population whose vectors are kept in registers.  Measured (registers / staged): average,
// fp32, N = 3 78 / 82 us, N = 10 162 / 164, N = 20 (ResNet-18) 136 / 139; EMA, fp32, N = 5 71 / 74, N = 10 309 / 313, 131072 coordinates of
// N = 16 4.6 / 6.1, N = 32 equal; EMA, bf16, 2^25 coordinates N = 2 49 / 59, ResNet-50
// N = 5 94 / 87, N = 8 156 / 133 (few resident warps); PAPA-all, bf16, N = 8 129 / 132; average, bf16, 3 * 2^23 coordinates, fp32 out N = 26 200 us in
// registers, 28 275, 32 293, 33 253 staged.
template <class T>
constexpr int regs_max_models(int op) { return op == kOpAverage ? (T::kBytes == 4 ? 32 : 26) : (T::kBytes == 4 ? 16 : (op == kOpEma ? 3 : 8)); }

template <class T, class TOUT, int OP, int N>
cudaError_t launch_regs_n(const ReduceArgs &args, uint64_t units, const LaunchShape &shape, cudaStream_t stream)
{
    if constexpr (N < regs_max_models<T>(OP))
        if (args.pop.N > N) return launch_regs_n<T, TOUT, OP, N + 1>(args, units, shape, stream);
    const unsigned threads = shape.threads > 0 ? static_cast<unsigned>(shape.threads) : 256u;
    const uint64_t grid = (units + threads - 1) / threads;
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    return launch_chained(regs_np_kernel<T, TOUT, OP, N>, static_cast<unsigned>(grid), threads, 0, stream, args);
}

// [P][N]: the populations that are kept in registers instead of staged.  Staging pays for copies that leave in 16-byte pieces of
// whole lines where a lane's registers would be read with gaps (N = 8: 128 bytes from lane to lane), and costs a trip
// through shared memory, which the bytes of a small group do not hide.  Staged / registers, 3 * 2^23 coordinates, fp32:
//   average  N = 2 60 / 44, 4 90 / 72, 6 127 / 102, 7 128 / 122, 8 137 / 185, 9 149 / 152, 10 178 / 169 us (bf16 out 4 89 / 65, 7 132 / 116)
//   EMA      N = 2 76 / 60, 4 133 / 128, 5 158 / 167, 8 238 / 402
//   PAPA-all N = 2 75 / 60, 3 91.3 / 90.9, 4 131 / 137
// bf16, whose staged sums are carried from vector to vector from 9 models on (fp32 out / bf16 out):
//   average  N = 2 42 / 36 and 37 / 34, 3 39 / 40 and 34 / 36, 4 51 / 45 and 44 / 40, 6 68 / 57 and 61 / 51, 7 66 / 65, 8 82 / 98 and 86 / 96, 9 115 / 83 and
//            136 / 76, 10 117 / 92 and 136 / 85, 12 122 / 112 and 134 / 108;  EMA N = 2 47 / 35, 3 57 / 67;  PAPA-all N = 2 44 / 32, 3 49 / 65
template <class T>
constexpr bool pn_in_registers(int op, int N)
{
    if (T::kBytes == 2) return op == kOpAverage ? N <= 12 && N != 3 && N != 8 : N == 2;
    return N <= (op == kOpAverage ? 7 : op == kOpEma ? 4 : 3);
}
constexpr int kPnRegsMax = 12;

template <class T, class TOUT, int OP, int N>
cudaError_t launch_regs_pn_n(const ReduceArgs &args, const LaunchShape &shape, cudaStream_t stream)
{
    if constexpr (N < kPnRegsMax)
        if (args.pop.N > N) return launch_regs_pn_n<T, TOUT, OP, N + 1>(args, shape, stream);
    if constexpr (pn_in_registers<T>(OP, N)) {
        const unsigned threads = shape.threads > 0 ? static_cast<unsigned>(shape.threads) : 256u;
        const uint64_t grid = (static_cast<uint64_t>(args.group_hi - args.group_lo) + threads - 1) / threads;
        if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
        return launch_chained(regs_pn_kernel<T, TOUT, OP, N>, static_cast<unsigned>(grid), threads, 0, stream, args);
    }
    return cudaErrorInvalidValue;   // pn_in_registers decided otherwise
}

template <class T, class TOUT, int OP>
cudaError_t launch_reduce_typed(const ReduceArgs &args, const LaunchShape &shape, cudaStream_t stream)
{
    const uint64_t units = args.group_hi > args.group_lo ? (args.group_hi - args.group_lo) / Unit<T>::kGroups : 0;
    if (units == 0) return cudaSuccess;
    const int N = args.pop.N;
    if (args.pop.layout == kLayoutPN) {
        if (pn_in_registers<T>(OP, N)) return launch_regs_pn_n<T, TOUT, OP, 2>(args, shape, stream);
        const int per_thread = units_per_thread(N);
        const size_t bytes = static_cast<size_t>(N | 1) * 16;
        if constexpr (Unit<T>::kElems == 8) {   // what pn_in_registers leaves of the populations below a vector's elements
            if (N == 3) return launch_dense(dense_pn_kernel<T, TOUT, OP, 3>, args, units, per_thread, bytes, shape, stream);
            if constexpr (OP != kOpAverage) switch (N) {
                case 4: return launch_dense(dense_pn_kernel<T, TOUT, OP, 4>, args, units, per_thread, bytes, shape, stream);
                case 5: return launch_dense(dense_pn_kernel<T, TOUT, OP, 5>, args, units, per_thread, bytes, shape, stream);
                case 6: return launch_dense(dense_pn_kernel<T, TOUT, OP, 6>, args, units, per_thread, bytes, shape, stream);
                case 7: return launch_dense(dense_pn_kernel<T, TOUT, OP, 7>, args, units, per_thread, bytes, shape, stream);
            }
        }
        return launch_dense(dense_pn_kernel<T, TOUT, OP, 0>, args, units, per_thread, bytes, shape, stream);
    }
    if (N <= regs_max_models<T>(OP)) return launch_regs_n<T, TOUT, OP, 2>(args, units, shape, stream);
    return launch_dense(staged_np_kernel<T, TOUT, OP>, args, units, units_per_thread(N), static_cast<size_t>(N) * 16, shape, stream);
}

}  // namespace wash
