// energy.cu -- E(z) of Eq. def_HUIO for a batch of states, and the sweep
// dispatcher.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "sa_internal.h"

namespace sa {

int launch_sweep_quio_i64(const SweepArgs&, int, int, bool, int, int, size_t, void*);
int launch_sweep_quio_f32(const SweepArgs&, int, int, bool, int, int, size_t, void*);
int launch_sweep_huio_i64(const SweepArgs&, int, int, bool, int, int, size_t, void*);
int launch_sweep_huio_f32(const SweepArgs&, int, int, bool, int, int, size_t, void*);

int launch_sweep(const SweepArgs& a, int zbytes, int rule, bool smem, int blocks, int threads, size_t shared_bytes,
                 void* stream) {
    if (a.m.kind == KIND_QUIO) {
        if (a.m.is_float) return launch_sweep_quio_f32(a, zbytes, rule, smem, blocks, threads, shared_bytes, stream);
        return launch_sweep_quio_i64(a, zbytes, rule, smem, blocks, threads, shared_bytes, stream);
    }
    if (a.m.is_float) return launch_sweep_huio_f32(a, zbytes, rule, smem, blocks, threads, shared_bytes, stream);
    return launch_sweep_huio_i64(a, zbytes, rule, smem, blocks, threads, shared_bytes, stream);
}

int launch_sliced_quio_i64(const SweepArgs&, int, int, int, int, size_t, void*, int*);
int launch_sliced_quio_f32(const SweepArgs&, int, int, int, int, size_t, void*, int*);
int launch_sliced_huio_i64(const SweepArgs&, int, int, int, int, size_t, void*, int*);
int launch_sliced_huio_f32(const SweepArgs&, int, int, int, int, size_t, void*, int*);

int launch_sweep_sliced(const SweepArgs& a, int zbytes, int rule, int grid, int threads, size_t shared_bytes,
                        void* stream, int* bps) {
    if (a.m.kind == KIND_QUIO) {
        if (a.m.is_float) return launch_sliced_quio_f32(a, zbytes, rule, grid, threads, shared_bytes, stream, bps);
        return launch_sliced_quio_i64(a, zbytes, rule, grid, threads, shared_bytes, stream, bps);
    }
    if (a.m.is_float) return launch_sliced_huio_f32(a, zbytes, rule, grid, threads, shared_bytes, stream, bps);
    return launch_sliced_huio_i64(a, zbytes, rule, grid, threads, shared_bytes, stream, bps);
}

int launch_batch_quio_i64(const BatchArgs&, int, int, bool, int, int, size_t, void*, bool);
int launch_batch_quio_f32(const BatchArgs&, int, int, bool, int, int, size_t, void*, bool);
int launch_batch_huio_i64(const BatchArgs&, int, int, bool, int, int, size_t, void*, bool);
int launch_batch_huio_f32(const BatchArgs&, int, int, bool, int, int, size_t, void*, bool);

int launch_batch(const BatchArgs& b, int is_float, int kind, int zbytes, int rule, bool smem, int blocks, int threads,
                 size_t shared_bytes, void* stream, bool set_attr) {
    if (kind == KIND_QUIO) {
        if (is_float) return launch_batch_quio_f32(b, zbytes, rule, smem, blocks, threads, shared_bytes, stream, set_attr);
        return launch_batch_quio_i64(b, zbytes, rule, smem, blocks, threads, shared_bytes, stream, set_attr);
    }
    if (is_float) return launch_batch_huio_f32(b, zbytes, rule, smem, blocks, threads, shared_bytes, stream, set_attr);
    return launch_batch_huio_i64(b, zbytes, rule, smem, blocks, threads, shared_bytes, stream, set_attr);
}

int sweep_max_shared_optin() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
}

namespace {

template <class T>
__device__ __forceinline__ T block_sum(T v, T* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    T tot = T(0);
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += red[i];
    return tot;
}

__device__ __forceinline__ long long ipow_ll(long long x, int e) {
    long long r = 1;
    for (int i = 0; i < e; ++i) r *= x;
    return r;
}
__device__ __forceinline__ double ipow_d(double x, int e) {
    double r = 1.0;
    for (int i = 0; i < e; ++i) r *= x;
    return r;
}

// One block per state.  QUIO: sum_k z_k (lin_k + diag_k z_k) + (1/2) sum over
// the symmetric adjacency.  HUIO: single-variable slots + interaction terms.
template <bool IS_FLOAT>
__global__ void __launch_bounds__(256) energy_kernel(const EnergyArgs a) {
    __shared__ long long red_i[8];
    __shared__ double red_d[8];
    const DevModel& m = a.m;
    const int64_t st = blockIdx.x;
    if (st >= a.n_states) return;
    const int32_t* z = a.states + st * (int64_t)m.n;
    long long e_i = 0, p_i = 0;
    double e_d = 0.0, p_d = 0.0;
    // bounds check: a value outside [l_k, u_k] is reported and not evaluated
    for (int k = threadIdx.x; k < m.n; k += blockDim.x) {
        const VarMeta mt = m.meta[k];
        const long long zk = z[k];
        if (zk < mt.lo || zk > (long long)mt.lo + (long long)mt.width) atomicExch(a.bad, 1);
    }
    if (m.kind == KIND_QUIO) {
        for (int k = threadIdx.x; k < m.n; k += blockDim.x) {
            const VarMeta mt = m.meta[k];
            long long zk = z[k];
            if (zk < mt.lo || zk > (long long)mt.lo + (long long)mt.width) continue;
            if (IS_FLOAT) {
                double f = 0.0;
                for (int e = mt.link_begin; e < mt.link_begin + mt.link_len; ++e)
                    f += (m.adj_d ? m.adj_d[e] : (double)m.adj_f[e]) * (double)z[m.adj_col[e]];
                e_d += (double)zk * (m.lin_d[k] + m.diag_d[k] * (double)zk);
                p_d += (double)zk * f;
            } else {
                long long f = 0;
                for (int e = mt.link_begin; e < mt.link_begin + mt.link_len; ++e) f += m.adj_i[e] * (long long)z[m.adj_col[e]];
                e_i += zk * (m.lin_i[k] + m.diag_i[k] * zk);
                p_i += zk * f;
            }
        }
    } else {
        for (int k = threadIdx.x; k < m.n; k += blockDim.x) {
            const VarMeta mt = m.meta[k];
            const long long zk = z[k];
            if (zk < mt.lo || zk > (long long)mt.lo + (long long)mt.width) continue;
            const int base = m.slot_base[k];
            uint64_t msk = m.omega[k] >> 1;
            int q = 0;
            long long pz = 1;
            double pzd = 1.0;
            while (msk) {
                pz *= zk;
                pzd *= (double)zk;
                if (msk & 1ull) {
                    if (IS_FLOAT) e_d += m.aconst_d[base + q] * pzd;
                    else e_i += m.aconst_i[base + q] * pz;
                    ++q;
                }
                msk >>= 1;
            }
        }
        for (int t = threadIdx.x; t < m.n_iterms; t += blockDim.x) {
            bool inb = true;
            if (IS_FLOAT) {
                double prod = m.tcoef_d[t];
                for (int p = m.term_ptr[t]; p < m.term_ptr[t + 1]; ++p) {
                    const int v = m.mem_var[p];
                    const VarMeta mv = m.meta[v];
                    if (z[v] < mv.lo || (long long)z[v] > (long long)mv.lo + (long long)mv.width) inb = false;
                    prod *= ipow_d((double)z[v], m.mem_exp[p]);
                }
                if (inb) e_d += prod;
            } else {
                long long prod = m.tcoef_i[t];
                for (int p = m.term_ptr[t]; p < m.term_ptr[t + 1]; ++p) {
                    const int v = m.mem_var[p];
                    const VarMeta mv = m.meta[v];
                    if (z[v] < mv.lo || (long long)z[v] > (long long)mv.lo + (long long)mv.width) inb = false;
                    prod *= ipow_ll((long long)z[v], m.mem_exp[p]);
                }
                if (inb) e_i += prod;
            }
        }
    }
    if (IS_FLOAT) {
        const double a1 = block_sum<double>(e_d, red_d);
        __syncthreads();
        const double a2 = block_sum<double>(p_d, red_d);
        if (threadIdx.x == 0) reinterpret_cast<double*>(a.energies)[st] = m.const_d + a1 + 0.5 * a2;
    } else {
        const long long a1 = block_sum<long long>(e_i, red_i);
        __syncthreads();
        const long long a2 = block_sum<long long>(p_i, red_i);
        if (threadIdx.x == 0) reinterpret_cast<long long*>(a.energies)[st] = m.const_i + a1 + a2 / 2;
    }
}

// ------------------------------------------------------------------ QUIO, several states per block
// E = sum_k z_k (lin_k + diag_k z_k + sum_{j > k} J_kj z_j): each pair once, from
// the row of its smaller variable (up_rec).  A block stages G states in shared
// memory, interleaved by variable and in 1, 2 or 4 bytes above z_base, so that
// one shared load gives z_j of all of them and a row's entries are read once per
// G states; a thread takes whole rows, four entries per vector load,
// rows of the same length and alignment side by side (an FP64 instruction holds
// the pipe for 16 cycles however few lanes want it).
// Sparse models with normal fp32 couplings and values within +-4095 take their
// pairs from a flat list instead (PAIRS): a row of eight entries leaves lanes of
// an FP64 instruction idle, and z_k z_j, a whole number below 2^24, is exact.
// What bounds it: FP64 multiply-adds (two lanes per cycle and SM), one per pair
// and state, 0.52 ms for 4096 states of 80,000 pairs (and 0.13 ms for the linear
// and square terms); the conversions to FP64, which share that pipe, are done by
// moving bits.  4096 states of 10,000 variables and 80,000 pairs, a call: one
// state per block from both ends of every pair 6.81 ms; by rows, four states per
// block, 1.91; from the list 1.76, and with no FP64 conversion left beside the
// bit moves (widen_normal) 0.82.
__device__ __forceinline__ double widen_f(float x) {
    const uint32_t u = __float_as_uint(x);
    const uint32_t e = (u >> 23) & 0xFFu;
    if (e - 1u >= 254u) return (double)x;   // zero, denormal, infinite, NaN
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
}
// The same for normal numbers and zeros alone, with no conversion beside it that
// a compiler could issue under a false predicate.
__device__ __forceinline__ double widen_normal(float x) {
    const uint32_t u = __float_as_uint(x);
    const uint32_t hi = (u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u);
    return __hiloint2double((u << 1) == 0u ? 0 : (int)hi, (int)(u << 29));
}
template <class Z>
__device__ __forceinline__ double widen_z(int z) {
    if constexpr (sizeof(Z) < 4) return widen_normal(__int2float_rn(z));   // (below 2^24: see launch_energy)
    else return __int2double_rn(z);
}

template <class Z, int G>
struct alignas(sizeof(Z) * G) ZPack {
    Z z[G];
};

template <bool IS_FLOAT, class Z, int G, bool PAIRS>
__global__ void __launch_bounds__(256) quio_energy_kernel(const EnergyArgs a) {
    using Acc = typename std::conditional<IS_FLOAT, double, long long>::type;
    extern __shared__ __align__(16) uint8_t zraw[];
    __shared__ Acc red[8];
    ZPack<Z, G>* zs = reinterpret_cast<ZPack<Z, G>*>(zraw);
    const DevModel& m = a.m;
    const int64_t s0 = (int64_t)blockIdx.x * G;
    const int ns = (int)min((int64_t)G, a.n_states - s0);
    // stage, with the bounds check: a value outside [l_k, u_k] is reported
    for (int k = threadIdx.x; k < m.n; k += blockDim.x) {
        const VarMeta mt = m.meta[k];
        ZPack<Z, G> q;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            long long zk = mt.lo;
            if (g < ns) {
                zk = a.states[(s0 + g) * m.n + k];
                if (zk < mt.lo || zk > (long long)mt.lo + (long long)mt.width) {
                    atomicExch(a.bad, 1);
                    zk = mt.lo;
                }
            }
            q.z[g] = (Z)(uint32_t)(zk - m.z_base);
        }
        zs[k] = q;
    }
    __syncthreads();
    Acc e[G];
#pragma unroll
    for (int g = 0; g < G; ++g) e[g] = Acc(0);
    if constexpr (PAIRS) {
        // z_k z_j is a whole number below 2^24: one conversion and one FP64
        // multiply-add per pair and state, in every lane
        constexpr int U = 4;
        const int2* pairs = reinterpret_cast<const int2*>(m.up_pair);
        for (int p0 = threadIdx.x; p0 < m.n_pairs; p0 += U * blockDim.x) {
            int2 q[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int p = p0 + u * (int)blockDim.x;
                q[u] = p < m.n_pairs ? __ldg(pairs + p) : make_int2(0, 0);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (p0 + u * (int)blockDim.x >= m.n_pairs) break;
                const ZPack<Z, G> zk = zs[q[u].x & 0xFFFF], zj = zs[(uint32_t)q[u].x >> 16];
                const double w = widen_normal(__int_as_float(q[u].y));
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int zz = (m.z_base + (int)zk.z[g]) * (m.z_base + (int)zj.z[g]);
                    e[g] = fma(w, widen_z<Z>(zz), e[g]);
                }
            }
        }
        for (int k = threadIdx.x; k < m.n; k += blockDim.x) {
            const double l = m.lin_d[k], d = m.diag_d[k];
            const ZPack<Z, G> zk = zs[k];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const double zd = widen_z<Z>(m.z_base + (int)zk.z[g]);
                e[g] += zd * (l + d * zd);
            }
        }
    } else {
        for (int i = threadIdx.x; i < m.n; i += blockDim.x) {
            const int4 rec = __ldg(reinterpret_cast<const int4*>(m.up_rec) + i);
            const int k = rec.x, first = rec.y, end = rec.z;
            Acc f[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if constexpr (IS_FLOAT) f[g] = m.lin_d[k];
                else f[g] = m.lin_i[k];
            }
            for (int q0 = first & ~3; q0 < end; q0 += 4) {
                const int4 c4 = __ldg(reinterpret_cast<const int4*>(m.adj_col + q0));
                const int col[4] = {c4.x, c4.y, c4.z, c4.w};
                Acc w[4];
                if constexpr (IS_FLOAT) {
                    if (m.adj_d != nullptr) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) w[u] = __ldg(m.adj_d + q0 + u);
                    } else {
                        const float4 w4 = __ldg(reinterpret_cast<const float4*>(m.adj_f + q0));
                        w[0] = widen_f(w4.x); w[1] = widen_f(w4.y); w[2] = widen_f(w4.z); w[3] = widen_f(w4.w);
                    }
                } else {
                    const longlong2* wp = reinterpret_cast<const longlong2*>(m.adj_i + q0);
                    const longlong2 wa = __ldg(wp), wb = __ldg(wp + 1);
                    w[0] = wa.x; w[1] = wa.y; w[2] = wb.x; w[3] = wb.y;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (q0 + u < first || q0 + u >= end) continue;
                    const ZPack<Z, G> zj = zs[col[u]];
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const int z = m.z_base + (int)(uint32_t)zj.z[g];
                        if constexpr (IS_FLOAT) f[g] += w[u] * widen_z<Z>(z);
                        else f[g] += w[u] * (long long)z;
                    }
                }
            }
            const ZPack<Z, G> zk = zs[k];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int z = m.z_base + (int)(uint32_t)zk.z[g];
                if constexpr (IS_FLOAT) {
                    const double zd = widen_z<Z>(z);
                    e[g] += zd * (f[g] + m.diag_d[k] * zd);
                } else {
                    e[g] += (long long)z * (f[g] + m.diag_i[k] * (long long)z);
                }
            }
        }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const Acc tot = block_sum<Acc>(e[g], red);
        if (threadIdx.x == 0 && g < ns) {
            if constexpr (IS_FLOAT) reinterpret_cast<double*>(a.energies)[s0 + g] = m.const_d + tot;
            else reinterpret_cast<long long*>(a.energies)[s0 + g] = m.const_i + tot;
        }
        __syncthreads();
    }
}

// Dynamic shared memory that a block may have beside its reduction scratch.
size_t energy_room() { return (size_t)sweep_max_shared_optin() - 1024; }

template <bool IS_FLOAT, class Z, int G, bool PAIRS>
int launch_quio_energy(const EnergyArgs& a, cudaStream_t st) {
    auto kern = quio_energy_kernel<IS_FLOAT, Z, G, PAIRS>;
    const size_t sh = (size_t)a.m.n * sizeof(Z) * G;
    // what a launch may use without a limit of its own, 48 KB, counts static and
    // dynamic bytes; the limit is the same for every call: one of a call's size could
    // be lowered by another thread's call before the launch
    if (sh > 47 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)energy_room());
        if (e != cudaSuccess) return (int)e;
    }
    kern<<<(unsigned)((a.n_states + G - 1) / G), 256, sh, st>>>(a);
    return (int)cudaGetLastError();
}

template <bool IS_FLOAT, class Z, int G>
int launch_quio_form(const EnergyArgs& a, cudaStream_t st) {
    if constexpr (IS_FLOAT && sizeof(Z) < 4)
        if (a.m.up_pair != nullptr) return launch_quio_energy<IS_FLOAT, Z, G, true>(a, st);
    return launch_quio_energy<IS_FLOAT, Z, G, false>(a, st);
}

// Four states per block when that still gives every SM two blocks and they
// fit, else one; returns false when one state does not fit on chip.
template <bool IS_FLOAT, class Z>
bool quio_energy_shape(const EnergyArgs& a, cudaStream_t st, int& rc) {
    const size_t room = energy_room(), one = (size_t)a.m.n * sizeof(Z);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (4 * one <= room && a.n_states >= 4 * 2 * (int64_t)sms) rc = launch_quio_form<IS_FLOAT, Z, 4>(a, st);
    else if (one <= room) rc = launch_quio_form<IS_FLOAT, Z, 1>(a, st);
    else return false;
    return true;
}
template <bool IS_FLOAT>
bool quio_energy(const EnergyArgs& a, cudaStream_t st, int& rc) {
    const uint32_t span = a.m.z_span;
    const long long lo = a.m.z_base, hi = lo + (long long)span;
    const bool small = lo > -(1 << 24) && hi < (1 << 24);   // exact in fp32 on the way to FP64
    if (small && span <= 0xFFu) return quio_energy_shape<IS_FLOAT, uint8_t>(a, st, rc);
    if (small && span <= 0xFFFFu) return quio_energy_shape<IS_FLOAT, uint16_t>(a, st, rc);
    return quio_energy_shape<IS_FLOAT, uint32_t>(a, st, rc);
}

}  // namespace

int launch_energy(const EnergyArgs& a, void* stream) {
    if (a.n_states <= 0) return 0;
    if (a.m.kind == KIND_QUIO) {
        int rc = 0;
        const bool done = a.m.is_float ? quio_energy<true>(a, (cudaStream_t)stream, rc)
                                       : quio_energy<false>(a, (cudaStream_t)stream, rc);
        if (done) return rc;
    }
    const unsigned grid = (unsigned)a.n_states;
    if (a.m.is_float) energy_kernel<true><<<grid, 256, 0, (cudaStream_t)stream>>>(a);
    else energy_kernel<false><<<grid, 256, 0, (cudaStream_t)stream>>>(a);
    return (int)cudaGetLastError();
}

}  // namespace sa
