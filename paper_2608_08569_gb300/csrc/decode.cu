// Stage-2 decode step of VoxZip for fp32 caches (and for shapes outside the tensor-core kernel's
// limits): cache append (Eq. 1), GQA attention (Eq. 2) and the temporally decayed accumulated score
// (Eq. 6), fused so that every cached K and V row is read once.
//
// One thread-block cluster of S CTAs per (layer, sequence, kv-head) unit; CTA r of the cluster
// owns the contiguous token range [r*ceil(n/S), (r+1)*ceil(n/S)). Per CTA:
//   1. its K and V rows are requested into L2; the CTA owning slot n (the new token) appends k_new,
//      v_new and its position;
//   2. K: a row per group of D/4 lanes, the group's queries in registers (GP heads, 2 to 16). The GP
//      dot products of a row are summed over the lanes by halves (9 shuffles for 8 heads and 32 lanes,
//      where a full sum of each takes 40), which leaves each lane one head's logit;
//   3. p = 2^(logit - the CTA's maximum) in shared memory, and its sum per head;
//   4. V: every warp takes its share of the rows for all heads, so a row is loaded once;
//   5. one exchange through distributed shared memory gives the unit's maximum and normaliser: the CTA
//      rewrites the scores of its tokens as gamma * s + sum_h p_h / Z_h and combines one slice of the
//      G x D outputs from all CTAs' partials.
// The products are fp32 on the CUDA cores throughout. At 192 units of 417 rows (84.6 MB, the 10-min
// 20x cache in fp32) this takes 20.5 us a launch; the kernel before it (every head's warp reading all of
// V, two exchanges, nothing ahead of the loads) took 75.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"
#include "evict_policy.cuh"
#include "ptx.cuh"

namespace cg = cooperative_groups;

namespace voxzip {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kTargetTokensPerCta = 256;  // tokens per CTA when the units fill the GPU,
constexpr int kFewTokensPerCta = 64;      // and when they do not: shorter ranges on more SMs
constexpr int kMaxCluster = 16;
constexpr size_t kMaxSmem = 227 * 1024;
constexpr int kRowBatch = 4;              // rows whose loads a lane has in flight

struct DecodeParams {
    const void *q, *k_new, *v_new;
    const int32_t *new_pos;
    void *k_cache, *v_cache;
    float *score;
    int32_t *pos, *len;
    void *out;
    int32_t *status;
    int32_t B, L, Hq, Hkv, G, C, layer_begin, chunk_cap;
    float gamma, scale_log2;
};

// Shared memory of a CTA: partial outputs [sets][heads][D], statistics [..][heads], logits [cap][heads],
// old scores [cap]. Long ranges (kBig) keep one set of partial outputs, which the warps add to in turn,
// no padding heads and no old scores, so that every length fits that fits beside two sets of outputs.
template <int D, int GP, bool kBig>
struct Smem {
    static constexpr int kStats = 2 * kWarps + 2 + kMaxCluster + 1;
    static size_t bytes(int G, int cap) {
        const size_t heads = kBig ? G : GP;
        return sizeof(float) * ((kBig ? 1 : kWarps) * heads * D + kStats * heads + cap * heads + (kBig ? 0 : cap));
    }
};

// GP: the group's heads, padded to 2, 4, 8 or 16. kBig: ranges too long for the roomier layout.
template <typename T, int D, int GP, bool kBig>
__global__ void __launch_bounds__(kThreads) decode_kernel(const DecodeParams p) {
    constexpr int kLanesPerRow = D / 4;           // lanes covering one row, 4 elements each
    constexpr int kRowsPerWarp = 32 / kLanesPerRow;
    constexpr int kRowStep = kWarps * kRowsPerWarp;

    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = p.G;

    extern __shared__ __align__(16) float smem[];
    const int H = kBig ? G : GP;             // heads kept
    float *ow = smem;                        // [warps][H][D]; the sum over warps lands in warp 0's
    float *m_w = ow + (kBig ? 1 : kWarps) * H * D;  // [warps][H] maxima
    float *z_w = m_w + kWarps * H;           // [warps][H] sums
    float *m_cta = z_w + kWarps * H, *z_cta = m_cta + H;
    float *fac = z_cta + H;                  // [S][H]: 2^(m_r - m) / Z; then this CTA's own
    float *fac_own = fac + kMaxCluster * H;
    float *lg = fac_own + H;                 // [chunk_cap][H] logits, then p
    float *s_old = lg + (size_t)p.chunk_cap * H;

    const UnitIdx ui = unit_of(blockIdx.y, p.B, p.L, p.Hkv, p.layer_begin);
    ptx::grid_dependency_wait();  // a programmatic dependent of the previous kernel: wait for its writes
    const int32_t n_old = p.len[ui.cache_unit];
    const int32_t n = n_old + 1;
    if (n_old < 0 || n > p.C) {  // same decision in every CTA of the cluster
        if (rank == 0 && tid == 0) raise_status(p.status, VOXZIP_DEV_CAPACITY);
        return;
    }
    const int chunk = (n + S - 1) / S;
    if (chunk > p.chunk_cap) {
        if (rank == 0 && tid == 0) raise_status(p.status, VOXZIP_DEV_LEN_HINT);
        return;
    }
    const int j0 = min(n, rank * chunk), j1 = min(n, j0 + chunk), cnt = j1 - j0;

    const int64_t act_row = (int64_t)ui.l_local * p.B + ui.b;   // [layer_local][B] activation row
    T *kc = static_cast<T *>(p.k_cache) + (ui.cache_unit * p.C + j0) * D;  // row 0 of the range
    T *vc = static_cast<T *>(p.v_cache) + (ui.cache_unit * p.C + j0) * D;
    float *sc = p.score + ui.cache_unit * p.C + j0;

    if (tid == 0 && cnt > 0) {
        ptx::prefetch_l2(kc, (uint32_t)cnt * D * sizeof(T));
        ptx::prefetch_l2(vc, (uint32_t)cnt * D * sizeof(T));
    }
    // Eq. 1: the CTA that owns slot n-1 appends the new token.
    const int jn = n - 1 - j0;
    if (jn >= 0 && jn < cnt) {
        const T *kn = static_cast<const T *>(p.k_new) + (act_row * p.Hkv + ui.h) * D;
        const T *vn = static_cast<const T *>(p.v_new) + (act_row * p.Hkv + ui.h) * D;
        for (int i = tid; i < D; i += kThreads) {
            kc[(int64_t)jn * D + i] = kn[i];
            vc[(int64_t)jn * D + i] = vn[i];
        }
        if (tid == 0) p.pos[ui.cache_unit * p.C + n - 1] = p.new_pos[ui.b];
    }
    // The old scores travel to shared memory while the rows stream.
    if constexpr (!kBig)
        for (int i = tid; i < cnt; i += kThreads)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(ptx::smem_u32(s_old + i)), "l"(sc + i)
                         : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int sub = lane / kLanesPerRow, e = (lane % kLanesPerRow) * 4;
    float4 q4[GP];
#pragma unroll
    for (int g = 0; g < GP; ++g) {
        q4[g] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (g < G) {
            const float4 x = load4(static_cast<const T *>(p.q) + (act_row * p.Hq + (int64_t)ui.h * G + g) * D + e);
            q4[g] = make_float4(x.x * p.scale_log2, x.y * p.scale_log2, x.z * p.scale_log2, x.w * p.scale_log2);
        }
    }
    __syncthreads();  // the appended row is visible

    // Logits for this CTA's tokens (Eq. 2 numerator), log2 domain. After the sum by halves a lane holds
    // head `head` of its row; one lane of those that hold the same value writes it.
    int head = 0;
#pragma unroll
    for (int o = kLanesPerRow / 2, w = GP / 2; w > 0; o >>= 1, w >>= 1) head += (lane & o) ? w : 0;
    const bool writer = (lane & (kLanesPerRow / GP - 1)) == 0 && head < H;
    float m = -INFINITY;
    for (int base = warp * kRowsPerWarp + sub; base - sub < cnt; base += kRowBatch * kRowStep) {
        float4 k4[kRowBatch];
#pragma unroll
        for (int u = 0; u < kRowBatch; ++u) {
            const int j = base + u * kRowStep;
            k4[u] = j < cnt ? load4(kc + (int64_t)j * D + e) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < kRowBatch; ++u) {
            const int j = base + u * kRowStep;
            if (j - sub >= cnt) break;  // the same decision in every lane
            float a[GP];
#pragma unroll
            for (int g = 0; g < GP; ++g)
                a[g] = q4[g].x * k4[u].x + q4[g].y * k4[u].y + q4[g].z * k4[u].z + q4[g].w * k4[u].w;
#pragma unroll
            for (int o = kLanesPerRow / 2, w = GP / 2; o > 0; o >>= 1, w >>= 1) {
                if (w > 0) {
                    const bool up = lane & o;
#pragma unroll
                    for (int g = 0; g < w; ++g) {
                        const float give = up ? a[g] : a[g + w], keep = up ? a[g + w] : a[g];
                        a[g] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
                } else {
                    a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
                }
            }
            if (j < cnt) {
                if (writer) lg[j * H + head] = a[0];
                m = fmaxf(m, a[0]);
            }
        }
    }
    if (kRowsPerWarp > 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    if (writer && sub == 0) m_w[warp * H + head] = m;
    __syncthreads();

    // p relative to the CTA's maximum (a maximum of -inf, from logits all -inf, counts as 0), and its sums.
    auto cta_max = [&](int g) {
        float mc = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) mc = fmaxf(mc, m_w[w * H + g]);
        return mc;
    };
    if (tid < H) m_cta[tid] = cta_max(tid);
    if constexpr (kBig) {
        for (int g = warp; g < H; g += kWarps) {
            const float mc = cta_max(g), mm = mc == -INFINITY ? 0.f : mc;
            float z = 0.f;
            for (int i = lane; i < cnt; i += 32) z += lg[i * H + g] = exp2f(lg[i * H + g] - mm);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
            if (lane < kWarps) z_w[lane * H + g] = lane == 0 ? z : 0.f;
        }
    } else {
        const float mc = cta_max(tid % GP), mm = mc == -INFINITY ? 0.f : mc;
        float z = 0.f;
        for (int i = tid; i < cnt * GP; i += kThreads) {  // i % GP stays the same
            const float x = exp2f(lg[i] - mm);
            lg[i] = x;
            z += x;
        }
#pragma unroll
        for (int o = 16; o >= GP; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        if (lane < GP) z_w[warp * GP + lane] = z;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // this thread's old scores have landed
    __syncthreads();

    // Partial P V over this CTA's tokens.
    {
        float4 o4[GP];
#pragma unroll
        for (int g = 0; g < GP; ++g) o4[g] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int base = warp * kRowsPerWarp + sub; base < cnt; base += kRowBatch * kRowStep) {
            float4 v4[kRowBatch];
#pragma unroll
            for (int u = 0; u < kRowBatch; ++u) {
                const int j = base + u * kRowStep;
                v4[u] = j < cnt ? load4(vc + (int64_t)j * D + e) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < kRowBatch; ++u) {
                const int j = base + u * kRowStep;
                if (j >= cnt) break;
                float pr[GP];
                if constexpr (kBig) {
#pragma unroll
                    for (int g = 0; g < GP; ++g) pr[g] = g < G ? lg[j * H + g] : 0.f;
                } else if constexpr (GP == 2) {
                    const float2 x = *reinterpret_cast<const float2 *>(lg + j * GP);
                    pr[0] = x.x, pr[1] = x.y;
                } else {
#pragma unroll
                    for (int g = 0; g < GP; g += 4) {
                        const float4 x = *reinterpret_cast<const float4 *>(lg + j * GP + g);
                        pr[g] = x.x, pr[g + 1] = x.y, pr[g + 2] = x.z, pr[g + 3] = x.w;
                    }
                }
#pragma unroll
                for (int g = 0; g < GP; ++g) {
                    o4[g].x += pr[g] * v4[u].x, o4[g].y += pr[g] * v4[u].y;
                    o4[g].z += pr[g] * v4[u].z, o4[g].w += pr[g] * v4[u].w;
                }
            }
        }
        if constexpr (kRowsPerWarp > 1) {
#pragma unroll
            for (int g = 0; g < GP; ++g) {
                o4[g].x += __shfl_xor_sync(0xffffffffu, o4[g].x, 16);
                o4[g].y += __shfl_xor_sync(0xffffffffu, o4[g].y, 16);
                o4[g].z += __shfl_xor_sync(0xffffffffu, o4[g].z, 16);
                o4[g].w += __shfl_xor_sync(0xffffffffu, o4[g].w, 16);
            }
        }
        if constexpr (kBig) {
            for (int w = 0; w < kWarps; ++w) {
                if (warp == w && sub == 0) {
#pragma unroll
                    for (int g = 0; g < GP; ++g)
                        if (g < G) {
                            float4 *o = reinterpret_cast<float4 *>(ow + g * D + e);
                            const float4 y = w > 0 ? *o : make_float4(0.f, 0.f, 0.f, 0.f);
                            *o = make_float4(y.x + o4[g].x, y.y + o4[g].y, y.z + o4[g].z, y.w + o4[g].w);
                        }
                }
                __syncthreads();
            }
        } else if (sub == 0) {
#pragma unroll
            for (int g = 0; g < GP; ++g) *reinterpret_cast<float4 *>(ow + (warp * GP + g) * D + e) = o4[g];
        }
    }
    ptx::launch_dependents();  // streaming is over: the next launch may begin its prologue
    if (tid < H) {
        float z = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) z += z_w[w * H + tid];
        z_cta[tid] = z;
    }
    __syncthreads();
    for (int i = tid * 4; i < (kBig ? 0 : GP * D); i += kThreads * 4) {
        float4 v = *reinterpret_cast<const float4 *>(ow + i);
#pragma unroll
        for (int w = 1; w < kWarps; ++w) {
            const float4 x = *reinterpret_cast<const float4 *>(ow + w * GP * D + i);
            v.x += x.x, v.y += x.y, v.z += x.z, v.w += x.w;
        }
        *reinterpret_cast<float4 *>(ow + i) = v;
    }
    cluster.sync();  // every CTA's m_cta, z_cta and summed outputs are final
    // CTA r writes slice r of the G x D outputs. For a cluster of SS CTAs all the partials of this
    // thread's elements are requested before the statistics, so the reads take one round trip.
    auto combine = [&](auto ss_tag) {
        constexpr int SS = decltype(ss_tag)::value;
        constexpr int E = (GP * D / SS + kThreads - 1) / kThreads;
        const int total = G * D, per = (total + SS - 1) / SS;
        const int lo = rank * per, hi = min(total, lo + per);
        float part[E][SS];
#pragma unroll
        for (int x = 0; x < E; ++x) {
            const int i = lo + tid + x * kThreads;
#pragma unroll
            for (int r = 0; r < SS; ++r) part[x][r] = i < hi ? *cluster.map_shared_rank(&ow[i], r) : 0.f;
        }
        if (tid < H) {
            float mr[SS], zr[SS], mx = -INFINITY, z = 0.f;
#pragma unroll
            for (int r = 0; r < SS; ++r) {
                mr[r] = *cluster.map_shared_rank(&m_cta[tid], r);
                zr[r] = *cluster.map_shared_rank(&z_cta[tid], r);
                mx = fmaxf(mx, mr[r]);
            }
#pragma unroll
            for (int r = 0; r < SS; ++r) {
                mr[r] = mr[r] == -INFINITY ? 0.f : exp2f(mr[r] - mx);
                z += mr[r] * zr[r];
            }
            const float rz = tid < G ? 1.f / z : 0.f;
#pragma unroll
            for (int r = 0; r < SS; ++r) {
                fac[r * H + tid] = mr[r] * rz;
                if (r == rank) fac_own[tid] = mr[r] * rz;
            }
        }
        __syncthreads();
        T *og = static_cast<T *>(p.out) + (act_row * p.Hq + (int64_t)ui.h * G) * D;
#pragma unroll
        for (int x = 0; x < E; ++x) {
            const int i = lo + tid + x * kThreads;
            if (i < hi) {
                float o = 0.f;
#pragma unroll
                for (int r = 0; r < SS; ++r) o += fac[r * H + i / D] * part[x][r];
                og[i] = Elem<T>::from_f(o);
            }
        }
    };
    switch (S) {
        case 1: combine(std::integral_constant<int, 1>{}); break;
        case 2: combine(std::integral_constant<int, 2>{}); break;
        case 4: combine(std::integral_constant<int, 4>{}); break;
        case 8: combine(std::integral_constant<int, 8>{}); break;
        default: combine(std::integral_constant<int, 16>{}); break;
    }
    // Done reading the peers' shared memory (every value has been used above); the score update touches
    // this CTA's own only.
    ptx::cluster_arrive_relaxed();
    // Eq. 6: A = gamma * [A, 0] + sum over the group's heads of the softmax.
    for (int i = tid; i < cnt; i += kThreads) {
        float add = 0.f;
#pragma unroll
        for (int g = 0; g < GP; ++g)
            if (!kBig || g < G) add += lg[i * H + g] * fac_own[g];
        sc[i] = i == jn ? add : p.gamma * (kBig ? sc[i] : s_old[i]) + add;
    }
    if (rank == 0 && tid == 0) p.len[ui.cache_unit] = n;
    // No CTA leaves while others may still read its shared memory.
    ptx::cluster_wait();
}

template <typename T, int D, int GP, bool kBig>
cudaError_t launch_t(const DecodeParams &prm, int S, int units, cudaStream_t stream) {
    auto kern = decode_kernel<T, D, GP, kBig>;
    static std::atomic<uint64_t> configured{0};
    const cudaError_t set = once_per_device(configured, [&] {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
        return e != cudaSuccess ? e : cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    });
    if (set != cudaSuccess) return set;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)S, (unsigned)units, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = Smem<D, GP, kBig>::bytes(prm.G, prm.chunk_cap);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // overlap the previous kernel's tail
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t err = cudaLaunchKernelEx(&cfg, kern, prm);
    if (err == cudaErrorNotSupported || err == cudaErrorInvalidValue) {  // no programmatic launch here
        cudaGetLastError();
        cfg.numAttrs = 1;
        err = cudaLaunchKernelEx(&cfg, kern, prm);
    }
    return err;
}

// f(T(), D, GP as integral constants) for the runtime shape.
template <typename T, int D, typename F>
auto dispatch_group(int G, F &&f) {
    if (G <= 2) return f(T(), std::integral_constant<int, D>{}, std::integral_constant<int, 2>{});
    if (G <= 4) return f(T(), std::integral_constant<int, D>{}, std::integral_constant<int, 4>{});
    if (G <= 8) return f(T(), std::integral_constant<int, D>{}, std::integral_constant<int, 8>{});
    return f(T(), std::integral_constant<int, D>{}, std::integral_constant<int, 16>{});
}
template <typename F>
auto dispatch(const voxzip_cache_desc &d, F &&f) {
    const int G = d.q_heads / d.kv_heads;
    if (d.head_dim == 128)
        return d.dtype == VOXZIP_BF16 ? dispatch_group<__nv_bfloat16, 128>(G, f) : dispatch_group<float, 128>(G, f);
    return d.dtype == VOXZIP_BF16 ? dispatch_group<__nv_bfloat16, 64>(G, f) : dispatch_group<float, 64>(G, f);
}

}  // namespace

cudaError_t launch_decode(const voxzip_cache_desc &d, int32_t layer_begin, int32_t layer_count,
                          const void *q, const void *k_new, const void *v_new, const int32_t *new_pos,
                          void *k_cache, void *v_cache, float *score, int32_t *pos, int32_t *len,
                          float gamma, float sm_scale, int32_t max_len, void *out, int32_t *status,
                          cudaStream_t stream, bool *unsupported) {
    *unsupported = false;
    if (decode_mma_supported(d)) {
        cudaError_t e = launch_decode_mma(d, layer_begin, layer_count, q, k_new, v_new, new_pos, k_cache, v_cache,
                                          score, pos, len, gamma, sm_scale, max_len, out, status, stream,
                                          unsupported);
        if (!*unsupported) return e;
        *unsupported = false;  // shape outside the tensor-core kernel's limits: the generic kernel runs
    }
    const int G = d.q_heads / d.kv_heads;
    const int units = layer_count * d.batch * d.kv_heads;
    const int nmax = (max_len > 0 && max_len < d.capacity) ? max_len : d.capacity;
    // Enough CTAs for the GPU first, then ranges of up to kTargetTokensPerCta tokens.
    const int sms = sm_count();
    int S = 1;
    while (S < kMaxCluster && ((nmax + S - 1) / S > kTargetTokensPerCta ||
                               ((int64_t)units * S < sms && (nmax + S - 1) / S > kFewTokensPerCta)))
        S <<= 1;
    auto smem_for = [&](int s, bool big) {
        return dispatch(d, [&](auto, auto dd, auto gp) {
            constexpr int D = decltype(dd)::value, GP = decltype(gp)::value;
            const int cap = (nmax + s - 1) / s;
            return big ? Smem<D, GP, true>::bytes(G, cap) : Smem<D, GP, false>::bytes(G, cap);
        });
    };
    while (smem_for(S, false) > kMaxSmem && S < kMaxCluster) S <<= 1;
    const bool big = smem_for(S, false) > kMaxSmem;
    if (big && smem_for(S, true) > kMaxSmem) {
        *unsupported = true;
        return cudaSuccess;
    }
    DecodeParams prm;
    prm.q = q; prm.k_new = k_new; prm.v_new = v_new; prm.new_pos = new_pos;
    prm.k_cache = k_cache; prm.v_cache = v_cache; prm.score = score; prm.pos = pos; prm.len = len;
    prm.out = out; prm.status = status;
    prm.B = d.batch; prm.L = d.layers; prm.Hq = d.q_heads; prm.Hkv = d.kv_heads; prm.G = G;
    prm.C = d.capacity; prm.layer_begin = layer_begin; prm.chunk_cap = (nmax + S - 1) / S;
    prm.gamma = gamma;
    const float scale = sm_scale > 0.f ? sm_scale : 1.0f / sqrtf((float)d.head_dim);
    prm.scale_log2 = scale * 1.4426950408889634f;  // log2(e): exp(x) = 2^(x log2 e)
    return dispatch(d, [&](auto t, auto dd, auto gp) {
        constexpr int D = decltype(dd)::value, GP = decltype(gp)::value;
        return big ? launch_t<decltype(t), D, GP, true>(prm, S, units, stream)
                   : launch_t<decltype(t), D, GP, false>(prm, S, units, stream);
    });
}

}  // namespace voxzip
