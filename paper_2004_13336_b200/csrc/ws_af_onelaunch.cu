// Adafactor for all shards as ONE kernel.
//
// Adafactor needs every row and column sum of g^2 before any element's update direction exists, and the
// direction's norm before any element can take its step (paper Section 4.1, reduces over sharded dimensions):
// three passes over a tensor.  As separate launches six kernels drain the GPU in turn.  Here the passes of every
// tensor are entries of one schedule, ordered so that a tensor's later passes run behind its first one while other
// tensors' first passes stream from DRAM.
//
//   P1  sum the R gradient copies of a block, keep the sum, add g^2 + eps to the row and column sums
//   M   the moving averages Rv', Cv' of a chunk of the factored state, 1/sqrt factors, sum of Rv'
//   P2  sums of w^2 and U^2 of a block
//   P3  w' = w - step size * U
//
// A block is a piece of the tensor's rows x cols matrix and not a run of its elements: a thread owns 8 columns
// and walks down the rows, the block's rows in parallel are summed in shared memory, and a column's sum takes one
// add to memory per block whatever the row length.  (One add per thread put all adds of a tall narrow matrix on a
// few addresses, where they follow one another: an encoder-decoder of 2.4 M parameters, 128 wide, took 118 us with
// one copy where the stages take 47, now 41; 0.86 M, 64 wide: 105, 56, 25 us.)  A row's sum needs one warp-wide
// reduction and one add per 256 columns.  Row lengths that 8 does not divide have 4 columns per thread, and those
// that 4 does not divide 4 scalar accesses in place of a vector one.
//
// What bounds it: on large models the bytes of three passes through DRAM, 4R + 24 per parameter, at the copy
// bandwidth (102 M parameters: 27.8, 39.7 and 55.9 bytes at R = 1, 4, 8, L2 hit rate 5 to 9 %).  The kept sums of
// the blocks in flight, 256 KB each on 444 resident CTAs, and the weights that P2 reads take the whole L2 before a
// later pass comes back to them, so that leaving them in L2 more firmly (evict-last hints, discarding them after
// P3) changed nothing.  On small models an entry's chain of dependent reads (ticket -> record -> tables and ready
// word -> data, then the arrival): hence large blocks and one record per entry.
// Measured against the six launches it replaces (us): Transformer set (211 M), fp32, R = 1 1148 -> 877, R = 4 1376 ->
// 1245, R = 8 1862 -> 1760; ResNet-50 set (25.6 M), R = 4 269 -> 164; 22.7 M parameters in ragged tensors, R = 2:
// 749 -> 166 (there a scalar reduction per element went to memory); 45 792 parameters, called from the host, 27 -> 15.5.
// The hand-over between the passes is a tiny model's whole time (P1 2.4, M 2.4, P2 2.0, its sum and step size 2.8, P3
// 1 us): a counter's fences are one, the step size is published before anything else is stored, its two roots are
// formed side by side, M reads the old state while it waits, and the rows in parallel are folded four at a time
// (24 K parameters 16.6 -> 15.1 us, 0.7 M 20.8 -> 19.0, 4.1 M 38.3 -> 36.8; ragged 172 -> 166).
//
// Tickets, waits and their progress argument are those of ws_onelaunch.cu: an entry waits only for entries with
// smaller tickets, which belong to CTAs that are running or have finished; every wait has an iteration limit.
#include "ws_kernels.cuh"

namespace wsk {
namespace {

constexpr int kSpinLimitAf = 1 << 22;

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" :: "l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ int ld_volatile_int(const int* p) {
    int v;
    asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// Position of element e of a tensor inside a packed [R][S] buffer.
__device__ __forceinline__ long long packed_pos(const WsAfTensor& T, long long e, long long S) {
    if (e < T.piece) return T.off + e;
    if ((((unsigned long long)e | (unsigned long long)T.piece) >> 32) == 0) {
        const unsigned r = (unsigned)e / (unsigned)T.piece;
        return r * S + T.off + ((unsigned)e - r * (unsigned)T.piece);
    }
    const long long r = e / T.piece;
    return r * S + T.off + (e - r * T.piece);
}

// A thread's W elements of one row.  WS_AF_VEC8: 8 consecutive ones as one 256-bit access, or (P.wide == 0) two
// quads 4 tpr columns apart, so that a warp's 128-bit accesses stay contiguous.  WS_AF_VEC4, WS_AF_FULL: 4
// consecutive ones.  WS_AF_SCALAR, WS_AF_NARROW: 4, tpr columns apart.  `mask` says which exist: all, or what the end of the
// row (scalar) or of the tensor (WS_AF_FULL) leaves.  Idx: their element offsets in a tensor (flat) or in a
// packed buffer.
template <int MODE>
struct Idx {
    static constexpr int W = ws_af_width(MODE);
    static constexpr int N = ws_af_scalar(MODE) ? 4 : MODE == WS_AF_VEC8 ? 2 : 1;
    long long i[N];
};
template <int MODE>
__device__ __forceinline__ Idx<MODE> index_of(const AfLaunch& P, const WsAfTensor& T, long long e, unsigned mask, int tpr, bool flat) {
    Idx<MODE> x;
    x.i[0] = flat ? e : packed_pos(T, e, P.S);             // (a piece starts on a multiple of 8 elements)
    if constexpr (MODE == WS_AF_VEC8) {
        if (P.wide) x.i[1] = x.i[0] + 4;
        else x.i[1] = flat ? e + 4 * tpr : packed_pos(T, e + 4 * tpr, P.S);
    } else if constexpr (ws_af_scalar(MODE)) {
#pragma unroll
        for (int j = 1; j < 4; ++j) {
            const long long ej = e + (long long)j * tpr;
            x.i[j] = flat ? ej : ((mask >> j) & 1u ? packed_pos(T, ej, P.S) : 0);
        }
    }
    return x;
}
// all W elements exist and can be moved as vectors
template <int MODE>
__device__ __forceinline__ bool whole(unsigned mask) {
    return MODE == WS_AF_VEC8 || MODE == WS_AF_VEC4 || (MODE == WS_AF_FULL && mask == 15u);
}
template <int MODE>
__device__ __forceinline__ long long at_of(const Idx<MODE>& x, int j) {
    return ws_af_scalar(MODE) ? x.i[j % Idx<MODE>::N] : x.i[0] + j;
}

template <bool GBF, int MODE>
__device__ __forceinline__ GradRaw<GBF, Idx<MODE>::W> load_grads(const void* base, const Idx<MODE>& x, unsigned mask, bool wide) {
    if constexpr (MODE == WS_AF_VEC8) {
        if (wide) return load_grad<GBF, 8>(base, x.i[0]);
        const GradRaw<GBF, 4> a = load_grad<GBF, 4>(base, x.i[0]), b = load_grad<GBF, 4>(base, x.i[1]);
        GradRaw<GBF, 8> g;
        if constexpr (GBF) {
            g.u = make_uint4(a.u.x, a.u.y, b.u.x, b.u.y);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) { g.f[j] = a.f[j]; g.f[4 + j] = b.f[j]; }
        }
        return g;
    } else if constexpr (!ws_af_scalar(MODE)) {
        if (whole<MODE>(mask)) return load_grad<GBF, 4>(base, x.i[0]);
        return load_grad_partial<GBF, 4>(base, x.i[0], __popc(mask));
    } else {
        GradRaw<GBF, 4> g;
        if constexpr (GBF) {
            const unsigned short* p = reinterpret_cast<const unsigned short*>(base);
            unsigned h[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) h[j] = (mask >> j) & 1u ? (unsigned)__ldcs(p + x.i[j]) : 0u;
            g.u = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
        } else {
            const float* p = reinterpret_cast<const float*>(base);
#pragma unroll
            for (int j = 0; j < 4; ++j) g.f[j] = (mask >> j) & 1u ? __ldcs(p + x.i[j]) : 0.f;
        }
        return g;
    }
}

// 8 floats that are read again (normal priority in L2) as one 256-bit access
__device__ __forceinline__ Fv<8> load8_keep(const float* p) {
    unsigned r[8];
    Fv<8> o;
    asm volatile("ld.global.L1::no_allocate.L2::evict_normal.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "l"(p));
#pragma unroll
    for (int i = 0; i < 8; ++i) o.f[i] = __uint_as_float(r[i]);
    return o;
}
// A thread's kept sums of one row (tpr: distance of its columns where they are kept element by element).
template <int MODE>
__device__ __forceinline__ Fv<Idx<MODE>::W> load_kept(const float* p, unsigned mask, int tpr) {
    if constexpr (MODE == WS_AF_VEC8) {
        return load8_keep(p);
    } else {
        Fv<4> o;
        if constexpr (MODE == WS_AF_NARROW) {
#pragma unroll
            for (int j = 0; j < 4; ++j) o.f[j] = (mask >> j) & 1u ? __ldcg(p + j * tpr) : 0.f;
        } else {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
            o.f[0] = v.x; o.f[1] = v.y; o.f[2] = v.z; o.f[3] = v.w;
        }
        return o;
    }
}
template <int MODE>
__device__ __forceinline__ void store_kept(float* p, const Fv<Idx<MODE>::W>& x, unsigned mask, int tpr) {
    if constexpr (MODE == WS_AF_VEC8) {
        store_f32<8>(p, x);
    } else if constexpr (MODE == WS_AF_NARROW) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((mask >> j) & 1u) __stcg(p + j * tpr, x.f[j]);
    } else {
        __stcg(reinterpret_cast<float4*>(p), make_float4(x.f[0], x.f[1], x.f[2], x.f[3]));
    }
}

// Weights: read at normal priority in P2 (P3 reads them again), streaming in P3.
template <int MODE, bool AGAIN>
__device__ __forceinline__ Fv<Idx<MODE>::W> load_weights(const float* p, const Idx<MODE>& x, unsigned mask, bool wide) {
    Fv<Idx<MODE>::W> o;
    if (MODE == WS_AF_VEC8 && wide) {
        if constexpr (MODE == WS_AF_VEC8) o = AGAIN ? load8_keep(p + x.i[0]) : load_f32<8>(p + x.i[0]);
    } else if (whole<MODE>(mask)) {
#pragma unroll
        for (int h = 0; h < Idx<MODE>::W / 4; ++h) {
            const float4* q = reinterpret_cast<const float4*>(p + x.i[h % Idx<MODE>::N]);
            const float4 v = AGAIN ? __ldcg(q) : __ldcs(q);
            o.f[4 * h] = v.x; o.f[4 * h + 1] = v.y; o.f[4 * h + 2] = v.z; o.f[4 * h + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float* q = p + at_of<MODE>(x, j);
            o.f[j] = (mask >> j) & 1u ? (AGAIN ? __ldcg(q) : __ldcs(q)) : 0.f;
        }
    }
    return o;
}
template <int MODE>
__device__ __forceinline__ void store_weights(float* p, const Idx<MODE>& x, unsigned mask, const Fv<Idx<MODE>::W>& w, bool wide) {
    if (MODE == WS_AF_VEC8 && wide) {
        if constexpr (MODE == WS_AF_VEC8) store_f32<8>(p + x.i[0], w);
    } else if (whole<MODE>(mask)) {
#pragma unroll
        for (int h = 0; h < Idx<MODE>::W / 4; ++h)
            __stcs(reinterpret_cast<float4*>(p + x.i[h % Idx<MODE>::N]), make_float4(w.f[4 * h], w.f[4 * h + 1], w.f[4 * h + 2], w.f[4 * h + 3]));
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((mask >> j) & 1u) p[at_of<MODE>(x, j)] = w.f[j];
    }
}
template <int MODE>
__device__ __forceinline__ void store_bf16s(unsigned short* p, const Idx<MODE>& x, unsigned mask, const Fv<Idx<MODE>::W>& w, bool wide) {
    if (MODE == WS_AF_VEC8 && wide) {
        if constexpr (MODE == WS_AF_VEC8) store_bf16<8>(p + x.i[0], w);
    } else if (whole<MODE>(mask)) {
#pragma unroll
        for (int h = 0; h < Idx<MODE>::W / 4; ++h) {
            Fv<4> q;
#pragma unroll
            for (int j = 0; j < 4; ++j) q.f[j] = w.f[4 * h + j];
            store_bf16<4>(p + x.i[h % Idx<MODE>::N], q);
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((mask >> j) & 1u) {
                const __nv_bfloat16 b = __float2bfloat16_rn(w.f[j]);
                p[at_of<MODE>(x, j)] = *reinterpret_cast<const unsigned short*>(&b);
            }
    }
}

// How a thread walks its block: nv vectors, the v-th of them in row rr + v * rp of the block, estep elements
// behind the one before.
struct Walk {
    int rr, c0;            // its row among the rp parallel ones, its first column in the block
    int nv;
    int passes;            // the block's largest nv (uniform)
    int kstep;             // floats between its kept vectors
    unsigned cmask;        // which of its columns exist
    long long e0, estep;   // first element, distance to the next vector's
    float* kept;           // vector v's kept sums are at kept + v * kstep
};
template <int MODE>
__device__ __forceinline__ Walk walk_of(const AfLaunch& P, const WsAfTensor& T, const WsAfItem& it) {
    constexpr int W = Idx<MODE>::W;
    Walk k;
    k.rr = (int)threadIdx.x / it.tpr;
    const int cc = (int)threadIdx.x - k.rr * it.tpr;
    k.c0 = ws_af_scalar(MODE) ? cc : (MODE == WS_AF_VEC8 && P.wide) ? 8 * cc : 4 * cc;
    k.passes = (it.nr + it.rp - 1) / it.rp;
    k.nv = (k.rr < it.rp && k.rr < it.nr) ? (it.nr - k.rr + it.rp - 1) / it.rp : 0;
    k.kstep = it.rp * ws_af_kept_row(MODE, it.nc, it.tpr);
    k.cmask = 15u;
    if (ws_af_scalar(MODE)) {
        k.cmask = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (cc + j * it.tpr < it.nc) k.cmask |= 1u << j;
    }
    k.e0 = ((long long)it.row0 + k.rr) * T.ncol + it.col0 + k.c0;
    k.estep = it.rp * T.ncol;
    k.kept = P.kept + (long long)it.goff32 * 32 + (MODE == WS_AF_NARROW ? k.rr * it.nc + cc : (int)threadIdx.x * W);
    return k;
}
template <int MODE>
__device__ __forceinline__ unsigned mask_of(const WsAfTensor& T, const Walk& k, int v, long long e) {
    if (v >= k.nv) return 0u;
    if (MODE != WS_AF_FULL) return k.cmask;
    const long long left = T.numel - e;
    return left >= 4 ? 15u : left <= 0 ? 0u : (1u << (int)left) - 1u;
}

// ------------------------------------------------------------------------ P1
// colsum: kBlock * W floats of shared memory.
template <bool GBF, int RB, int U, bool LOOPK, int MODE>
__device__ __forceinline__ void sums_block(const AfLaunch& P, const WsAfTensor& T, const WsAfItem& it, const void* const* sgp,
                                           float* colsum) {
    constexpr int W = Idx<MODE>::W;
    const bool wide = P.wide != 0;
    const Walk k = walk_of<MODE>(P, T, it);
    float cacc[W];
#pragma unroll
    for (int j = 0; j < W; ++j) cacc[j] = 0.f;
    // lanes that share a row are consecutive; bit i: lane + 2^i shares this lane's row
    const int lane = threadIdx.x & 31;
    unsigned same = 0;
    bool head = false;
    if (MODE != WS_AF_FULL) {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const int ro = __shfl_down_sync(0xffffffffu, k.rr, 1 << i);
            if (lane + (1 << i) < 32 && ro == k.rr) same |= 1u << i;
        }
        const int rp = __shfl_up_sync(0xffffffffu, k.rr, 1);
        head = lane == 0 || rp != k.rr;
    }
    float* rowacc = P.acc + T.irow + it.row0 + k.rr;
    long long e = k.e0;
    for (int v0 = 0; v0 < k.passes; v0 += U, e += U * k.estep) {
        unsigned m[U];
        Idx<MODE> x[U];
        Fv<W> g[U], comp[LOOPK ? U : 1];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            m[u] = mask_of<MODE>(T, k, v0 + u, e + u * k.estep);
            if (m[u]) x[u] = index_of<MODE>(P, T, e + u * k.estep, m[u], it.tpr, P.fused != 0);
        }
        for (int k0 = 0; k0 < (LOOPK ? P.R : 1); k0 += RB) {
            GradRaw<GBF, W> raw[U][RB];
#pragma unroll
            for (int j = 0; j < RB; ++j)
                if (RB == 1 || k0 + j < P.R) {
                    const void* gk = sgp[k0 + j];
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (m[u]) raw[u][j] = load_grads<GBF, MODE>(gk, x[u], m[u], wide);
                }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                Fv<W> gb[RB];
#pragma unroll
                for (int j = 0; j < RB; ++j) {
                    if ((RB == 1 || k0 + j < P.R) && m[u]) {
                        gb[j] = widen<GBF, W>(raw[u][j]);
                    } else {
#pragma unroll
                        for (int i = 0; i < W; ++i) gb[j].f[i] = 0.f;
                    }
                }
#pragma unroll
                for (int s = 1; s < RB; s <<= 1)
#pragma unroll
                    for (int j = 0; j + s < RB; j += 2 * s)
#pragma unroll
                        for (int i = 0; i < W; ++i) gb[j].f[i] += gb[j + s].f[i];
                if constexpr (!LOOPK) {
                    g[u] = gb[0];
                } else if (k0 == 0) {
                    g[u] = gb[0];
#pragma unroll
                    for (int i = 0; i < W; ++i) comp[u].f[i] = 0.f;
                } else {
#pragma unroll
                    for (int i = 0; i < W; ++i) kahan1(g[u].f[i], comp[u].f[i], gb[0].f[i]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float racc = 0.f;
            if (m[u]) {
                float q[W];
#pragma unroll
                for (int j = 0; j < W; ++j) {
                    g[u].f[j] *= P.gscale;
                    q[j] = fmaf(g[u].f[j], g[u].f[j], P.eps);
                    if (MODE == WS_AF_VEC8 || MODE == WS_AF_VEC4 || (m[u] >> j) & 1u) {
                        racc += q[j];
                        cacc[j] += q[j];
                    }
                }
                store_kept<MODE>(k.kept + (long long)(v0 + u) * k.kstep, g[u], m[u], it.tpr);
                if (MODE == WS_AF_FULL) {
                    // unfactored: the element's own second moment, final here
                    const long long eu = e + u * k.estep;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if ((m[u] >> j) & 1u) {
                            float* s = P.state + T.foff + eu + j;
                            const float nv = (float)(P.beta * (double)*s + (1.0 - P.beta) * (double)q[j]);
                            *s = nv;
                            P.fac[T.icol + eu + j] = (float)(1.0 / sqrt((double)nv));
                        }
                }
            }
            if (MODE != WS_AF_FULL) {
                // the row's sum over the lanes that share it, added to memory by the first of them
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const float y = __shfl_down_sync(0xffffffffu, racc, 1 << i);
                    if ((same >> i) & 1u) racc += y;
                }
                if (head && v0 + u < k.nv) atomicAdd(rowacc + (v0 + u) * it.rp, racc);
            }
        }
    }
    if constexpr (MODE != WS_AF_FULL) {
        // the block's rows in parallel are summed here first, so that a column's sum takes one add per block: adds
        // to one address follow one another, and a tall narrow matrix has all its adds on a few addresses
        int rows = it.rp < it.nr ? it.rp : it.nr;
        const int width = it.tpr * W;                     // columns, some of them beyond a row whose length 4 does not divide
        const int h = wide && MODE == WS_AF_VEC8 ? 4 : 4 * it.tpr;   // from a thread's first quad to its second
        if (rows > 1) {
            float* mine = colsum + k.rr * width + k.c0;
            if (k.nv > 0) {
                if constexpr (!ws_af_scalar(MODE)) {
                    *reinterpret_cast<float4*>(mine) = make_float4(cacc[0], cacc[1], cacc[2], cacc[3]);
                    if constexpr (W == 8) *reinterpret_cast<float4*>(mine + h) = make_float4(cacc[4], cacc[5], cacc[6], cacc[7]);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) mine[j * it.tpr] = cacc[j];
                }
            }
            const int quads = width / 4;
            while (rows > 1) {                            // fold the upper three quarters of the rows onto the lowest
                const int part = (rows + 3) / 4;
                __syncthreads();
                for (int i = threadIdx.x; i < part * quads; i += kBlock) {
                    float4* a = reinterpret_cast<float4*>(colsum) + i;
                    float4 s[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        s[j] = i + j * part * quads < rows * quads ? a[j * part * quads] : make_float4(0.f, 0.f, 0.f, 0.f);
                    *a = make_float4((s[0].x + s[1].x) + (s[2].x + s[3].x), (s[0].y + s[1].y) + (s[2].y + s[3].y),
                                     (s[0].z + s[1].z) + (s[2].z + s[3].z), (s[0].w + s[1].w) + (s[2].w + s[3].w));
                }
                rows = part;
            }
            __syncthreads();
            if (k.rr == 0 && k.nv > 0) {
                if constexpr (!ws_af_scalar(MODE)) {
                    const float4 a = *reinterpret_cast<const float4*>(mine);
                    cacc[0] = a.x; cacc[1] = a.y; cacc[2] = a.z; cacc[3] = a.w;
                    if constexpr (W == 8) {
                        const float4 b = *reinterpret_cast<const float4*>(mine + h);
                        cacc[4] = b.x; cacc[5] = b.y; cacc[6] = b.z; cacc[7] = b.w;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) cacc[j] = mine[j * it.tpr];
                }
            }
        }
        if (k.rr == 0 && k.nv > 0) {
            float* c = P.acc + T.icol + it.col0 + k.c0;
            if constexpr (!ws_af_scalar(MODE)) {
                red_add_vec<4>(c, cacc);
                if constexpr (W == 8) red_add_vec<4>(c + h, cacc + 4);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if ((k.cmask >> j) & 1u) atomicAdd(c + j * it.tpr, cacc[j]);
            }
        }
    }
}

// ------------------------------------------------------------------ P2 and P3
template <bool APPLY, int MODE>
__device__ __forceinline__ void second_block(const AfLaunch& P, const WsAfTensor& T, const WsAfItem& it, double rscale,
                                             float rate, char* wt, double& sw, double& su) {
    constexpr int W = Idx<MODE>::W;
    constexpr int U = MODE == WS_AF_VEC4 ? 4 : 2;
    const bool wide = P.wide != 0;
    const Walk k = walk_of<MODE>(P, T, it);
    float* wbase = P.master ? reinterpret_cast<float*>(wt) : P.w;
    // column factors: the same columns in every row of the block
    float fc[W];
#pragma unroll
    for (int j = 0; j < W; ++j) fc[j] = 0.f;
    if (MODE != WS_AF_FULL && k.nv > 0) {
        const float* c = P.fac + T.icol + it.col0 + k.c0;
        if constexpr (!ws_af_scalar(MODE)) {
#pragma unroll
            for (int h = 0; h < W / 4; ++h) {
                const float4 t = __ldcg(reinterpret_cast<const float4*>(c + (h == 0 ? 0 : wide ? 4 : 4 * it.tpr)));
                fc[4 * h] = t.x; fc[4 * h + 1] = t.y; fc[4 * h + 2] = t.z; fc[4 * h + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) fc[j] = (k.cmask >> j) & 1u ? __ldcg(c + j * it.tpr) : 0.f;
        }
    }
    // a row's factor sqrt(sum(Rv') / Rv'_i) is formed in 64 bits and rounded once, like the stages'
    const double* rowfac = P.rfac + T.rfac + it.row0 + k.rr;
    long long e = k.e0;
    for (int v0 = 0; v0 < k.passes; v0 += U, e += U * k.estep) {
        unsigned m[U];
        Idx<MODE> x[U];
        Fv<W> g[U], w[U];
        float4 fv[MODE == WS_AF_FULL ? U : 1];
        double fr[U];
        float tw = 0.f, tu = 0.f;      // of up to 16 elements; a block's thread walks over 256, which are summed in 64 bits
#pragma unroll
        for (int u = 0; u < U; ++u) {
            m[u] = mask_of<MODE>(T, k, v0 + u, e + u * k.estep);
            if (m[u]) {
                x[u] = index_of<MODE>(P, T, e + u * k.estep, m[u], it.tpr, P.master != 0);
                g[u] = load_kept<MODE>(k.kept + (long long)(v0 + u) * k.kstep, m[u], it.tpr);
                w[u] = load_weights<MODE, !APPLY>(wbase, x[u], m[u], wide);
                if constexpr (MODE == WS_AF_FULL) fv[u] = __ldcg(reinterpret_cast<const float4*>(P.fac + T.icol + e + u * k.estep));
                else fr[u] = __ldcg(rowfac + (v0 + u) * it.rp);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!m[u]) continue;
            float frs = 1.f;
            if constexpr (MODE == WS_AF_FULL) { fc[0] = fv[u].x; fc[1] = fv[u].y; fc[2] = fv[u].z; fc[3] = fv[u].w; }
            else frs = (float)(fr[u] * rscale);
#pragma unroll
            for (int j = 0; j < W; ++j) {
                if ((ws_af_scalar(MODE) || MODE == WS_AF_FULL) && !((m[u] >> j) & 1u)) continue;
                const float uu = (g[u].f[j] * frs) * fc[j];
                if (APPLY) {
                    w[u].f[j] = fmaf(-rate, uu, w[u].f[j]);
                } else {
                    tw = fmaf(w[u].f[j], w[u].f[j], tw);
                    tu = fmaf(uu, uu, tu);
                }
            }
            if constexpr (APPLY) {
                store_weights<MODE>(wbase, x[u], m[u], w[u], wide);
                if (P.out == O_F32 || P.out == O_BF16) {          // next to the sharded state
                    if (P.fused) x[u] = index_of<MODE>(P, T, e + u * k.estep, m[u], it.tpr, true);
                    char* dst = P.fused ? wt : reinterpret_cast<char*>(P.gathered);
                    if (P.out == O_F32) store_weights<MODE>(reinterpret_cast<float*>(dst), x[u], m[u], w[u], wide);
                    else store_bf16s<MODE>(reinterpret_cast<unsigned short*>(dst), x[u], m[u], w[u], wide);
                }
            }
        }
        if constexpr (!APPLY) {
            sw += (double)tw;
            su += (double)tu;
        }
    }
}

// The waits of an entry for what earlier entries set: a ready word (0 when the wait ran out), or a count.
__device__ __forceinline__ unsigned long long wait_word(const AfLaunch& P, const unsigned long long* p) {
    unsigned long long word = 0;
    for (int tries = 0; tries < kSpinLimitAf; ++tries) {
        word = ld_acquire64(p);
        if (word != 0) return word;
        if ((tries & 255) == 255 && ld_volatile_int(P.status) != 0) break;
        __nanosleep(50);
    }
    atomicExch(P.status, 1);          // gave up: the update stays incomplete, the caller can tell
    return 0;
}
__device__ __forceinline__ bool wait_count(const AfLaunch& P, const int* p, int n) {
    for (int tries = 0; tries < kSpinLimitAf; ++tries) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        if (v >= n) return true;
        if ((tries & 255) == 255 && ld_volatile_int(P.status) != 0) break;
        __nanosleep(50);
    }
    atomicExch(P.status, 1);
    return false;
}

// Writes the pads of tensor t's packed state and output (+0).
__device__ void zero_pads(const AfLaunch& P, const WsAfTensor& T) {
    const bool concat = T.piece >= (1LL << 60);
    const long long end = concat ? T.pad_end : (long long)P.nshards * T.piece;
    for (long long e = T.numel + threadIdx.x; e < end; e += kBlock) {
        const long long pos = packed_pos(T, e, P.S);
        P.w[pos] = 0.f;
        if (!P.fused) {
            if (P.out == O_F32) reinterpret_cast<float*>(P.gathered)[pos] = 0.f;
            else if (P.out == O_BF16) reinterpret_cast<unsigned short*>(P.gathered)[pos] = 0;
        }
    }
}

template <bool GBF, int RB, int U, bool LOOPK, int NP>
__global__ void __launch_bounds__(kBlock, kMinBlocks) af_kernel(const AfLaunch P, const __grid_constant__ GradPtrs<NP> gp) {
    __shared__ unsigned long long s_word;
    __shared__ const void* sgp[NP];
    __shared__ float s_rate;
    __shared__ __align__(16) float colsum[kBlock * 8];
    __shared__ double da[kBlock / 32], db[kBlock / 32];
    __shared__ int s_last;
    const int tid = threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");     // the counters are cleared by the kernel in front

    if (tid == 0) s_word = atomicAdd(P.ticket, 1ULL);
    __syncthreads();
    const unsigned long long tk = s_word;
    if (tk >= P.nsched) return;
    __syncthreads();
    if (tk == 0) {
        // tensors without any element take part in no entry
        for (int t = tid; t < P.T; t += kBlock)
            if (P.tensors[t].item_count == 0) {
                const float a = (float)(P.eps2 * P.rho_step);
                P.alpha[t] = a;
                P.rho[t] = a;
                P.norms[2 * t] = 0.0;
                P.norms[2 * t + 1] = 0.0;
            }
        // (the concatenated layout's tail belongs to the last tensor, which may be one of them)
        if (!P.master && P.tensors[P.T - 1].item_count == 0) zero_pads(P, P.tensors[P.T - 1]);
    }
    // one access for the record, then everything that it leads to side by side
    WsAfItem it;
    {
        const uint4* src = reinterpret_cast<const uint4*>(P.sched + tk);
        const uint4 a = __ldg(src), b = __ldg(src + 1);
        it.seg = (int)a.x; it.row0 = (int)a.y; it.col0 = (int)a.z; it.goff32 = a.w;
        it.nr = (unsigned short)(b.x & 0xffffu); it.nc = (unsigned short)(b.x >> 16);
        it.tpr = (unsigned short)(b.y & 0xffffu); it.rp = (unsigned short)(b.y >> 16);
        it.item = b.z; it.phase = (int)b.w;
    }
    const int kind = it.phase;
    const WsAfTensor T = P.tensors[it.seg];
    char* wt = nullptr;
    if (kind >= 2 && P.wtab) wt = reinterpret_cast<char*>(P.wtab[it.seg]);
    if (kind == 0)
        for (int j = tid; j < P.R; j += kBlock) sgp[j] = P.fused ? P.gtab[(long long)it.seg * P.R + j] : gp.p[j];

    if (kind == 1) {
        // moments of one chunk of a tensor's factored state
        const long long begin = (long long)(((unsigned long long)(unsigned)it.col0 << 32) | (unsigned)it.row0);
        constexpr int N = kWsAfChunk / kBlock;
        float old[N];                              // (does not depend on P1)
#pragma unroll
        for (int j = 0; j < N; ++j) old[j] = tid + j * kBlock < (int)it.goff32 ? P.state[T.foff + begin + tid + j * kBlock] : 0.f;
        if (tid == 0) s_last = wait_count(P, P.count1 + it.seg, T.item_count);
        __syncthreads();
        if (!s_last) return;
        double rs = 0.0;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int i = tid + j * kBlock;
            if (i >= (int)it.goff32) break;
            const long long e = begin + i;
            const bool isrow = e < T.nrow;
            const long long k = isrow ? T.irow + e : T.icol + (e - T.nrow);
            const double v = P.beta * (double)old[j] + (1.0 - P.beta) * (double)__ldcg(P.acc + k);
            P.state[T.foff + e] = (float)v;
            const double f = rsqrt((double)(float)v);
            if (isrow) P.rfac[T.rfac + e] = f;
            else P.fac[k] = (float)f;
            if (isrow) rs += v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, o);
        if ((tid & 31) == 0) da[tid >> 5] = rs;
        __syncthreads();
        if (tid == 0) {
            for (int i = 1; i < kBlock / 32; ++i) rs += da[i];
            if (rs != 0.0) atomicAdd(P.rsum + it.seg, rs);
            if (arrive(P.countm + it.seg) == T.chunk_count) {
                // the row factors still lack sqrt(sum(Rv')), which goes with the word
                // (its bits inverted: no square root gives the word 0)
                const double r = sqrt(__ldcg(P.rsum + it.seg));
                st_release64(P.flagm + it.seg, ~(unsigned long long)__double_as_longlong(r));
            }
        }
        return;
    }
#ifdef WS_DEBUG_BOUNDS
    {
        unsigned bits = 0;
        const long long last = T.nrow > 0 ? ((long long)it.row0 + it.nr - 1) * T.ncol + it.col0 + it.nc - 1 : T.numel - 1;
        if (last >= T.numel || it.col0 < 0 || it.row0 < 0) bits |= WS_BOUNDS_STATE;
        if (!P.master && packed_pos(T, last, P.S) >= P.state_elems) bits |= WS_BOUNDS_STATE;
        if (!P.fused && packed_pos(T, last, P.S) >= P.state_elems) bits |= WS_BOUNDS_GRAD;
        if ((long long)it.goff32 * 32 + (long long)it.nr * ws_af_kept_row(T.mode, it.nc, it.tpr) > P.kept_elems)
            bits |= WS_BOUNDS_OUT;
        if (bits && tid == 0 && P.bounds) atomicOr(P.bounds, bits);
        if (bits) return;
    }
#endif

    if (kind == 0) {
        __syncthreads();
        if (T.mode == WS_AF_VEC8) sums_block<GBF, RB, U, LOOPK, WS_AF_VEC8>(P, T, it, sgp, colsum);
        else if (T.mode == WS_AF_VEC4) sums_block<GBF, RB, U, LOOPK, WS_AF_VEC4>(P, T, it, sgp, colsum);
        else if (T.mode == WS_AF_SCALAR) sums_block<GBF, RB, U, LOOPK, WS_AF_SCALAR>(P, T, it, sgp, colsum);
        else if (T.mode == WS_AF_NARROW) sums_block<GBF, RB, U, LOOPK, WS_AF_NARROW>(P, T, it, sgp, colsum);
        else sums_block<GBF, RB, 1, LOOPK, WS_AF_FULL>(P, T, it, sgp, colsum);
        __syncthreads();
        // (no CTA looks whether it was the last one: M waits for the count, and this CTA is done at once)
        if (tid == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" :: "l"(P.count1 + it.seg) : "memory");
        return;
    }

    // a factored tensor's row factors lack sqrt(sum(Rv')), which comes with M's ready word; P3 also needs the rate
    if (tid == 0) {
        unsigned long long a = ~(unsigned long long)__double_as_longlong(1.0), b = 1ULL;
        if (kind == 3) b = wait_word(P, P.flag2 + it.seg);
        if (T.chunk_count > 0) a = wait_word(P, P.flagm + it.seg);
        else if (kind == 2 && !wait_count(P, P.count1 + it.seg, T.item_count)) a = 0;
        s_word = ~a;
        s_rate = __uint_as_float((unsigned)(b >> 32));
        s_last = (a && b) ? 1 : 0;
    }
    __syncthreads();
    if (!s_last) return;
    const double rscale = __longlong_as_double((long long)s_word);
    double sw = 0.0, su = 0.0;
    if (kind == 3) {
        const float rate = s_rate;
        if (T.mode == WS_AF_VEC8) second_block<true, WS_AF_VEC8>(P, T, it, rscale, rate, wt, sw, su);
        else if (T.mode == WS_AF_VEC4) second_block<true, WS_AF_VEC4>(P, T, it, rscale, rate, wt, sw, su);
        else if (T.mode == WS_AF_SCALAR) second_block<true, WS_AF_SCALAR>(P, T, it, rscale, rate, wt, sw, su);
        else if (T.mode == WS_AF_NARROW) second_block<true, WS_AF_NARROW>(P, T, it, rscale, rate, wt, sw, su);
        else second_block<true, WS_AF_FULL>(P, T, it, rscale, rate, wt, sw, su);
        return;
    }
    if (T.mode == WS_AF_VEC8) second_block<false, WS_AF_VEC8>(P, T, it, rscale, 0.f, wt, sw, su);
    else if (T.mode == WS_AF_VEC4) second_block<false, WS_AF_VEC4>(P, T, it, rscale, 0.f, wt, sw, su);
    else if (T.mode == WS_AF_SCALAR) second_block<false, WS_AF_SCALAR>(P, T, it, rscale, 0.f, wt, sw, su);
    else if (T.mode == WS_AF_NARROW) second_block<false, WS_AF_NARROW>(P, T, it, rscale, 0.f, wt, sw, su);
    else second_block<false, WS_AF_FULL>(P, T, it, rscale, 0.f, wt, sw, su);
    double a = sw, b = su;
    sum_block(a, b, da, db);
    if (tid == 0) {
        P.ipart[it.item] = make_double2(a, b);
        s_last = arrive(P.count2 + it.seg) == T.item_count ? 1 : 0;
    }
    __syncthreads();
    if (!s_last) return;
    a = 0.0;
    b = 0.0;
    for (int i = tid; i < T.item_count; i += kBlock) {     // fixed order
        const double2 p = __ldcg(P.ipart + T.item_first + i);
        a += p.x;
        b += p.y;
    }
    sum_block(a, b, da, db);
    if (tid < 32) {
        // (two lanes: a 64-bit root and quotient take longer than the exchange)
        const double b0 = __shfl_sync(0xffffffffu, b, 0), mine = tid == 0 ? a : b0;
        const double rms = sqrt(mine / (double)T.numel), rms_u = __shfl_down_sync(0xffffffffu, rms, 1);
        if (tid == 0) {
            const double al = (P.eps2 > rms ? P.eps2 : rms) * P.rho_step, d = rms_u / P.clip;
            const float rate = (float)(d > 1.0 ? al / d : al);
            // the word first: it is what the other CTAs wait for
            st_release64(P.flag2 + it.seg, ((unsigned long long)__float_as_uint(rate) << 32) | 1ULL);
            P.norms[2 * it.seg] = a;
            P.norms[2 * it.seg + 1] = b;
            P.alpha[it.seg] = (float)al;
            P.rho[it.seg] = rate;
        }
    }
    if (!P.master) zero_pads(P, T);
}

template <bool GBF, int RB, int U, bool LOOPK, int NP>
ws_status launch(const AfLaunch& P, const void* const* gptrs, cudaStream_t st) {
    GradPtrs<NP> gp;
    for (int k = 0; k < NP; ++k) gp.p[k] = (gptrs && k < P.R) ? gptrs[k] : nullptr;
    launch_pdl(af_kernel<GBF, RB, U, LOOPK, NP>, P.nsched, st, P, gp);
    return ws_check_launch("one-kernel Adafactor");
}

// Loads in flight per thread: RB copies x U rows of 32 bytes (16 with bf16 gradients or 4-column threads); more
// copies than 4 are summed 4 at a time, compensated.
template <bool GBF>
ws_status launch_r(const AfLaunch& P, const void* const* gptrs, cudaStream_t st) {
    if (P.R == 1) return launch<GBF, 1, 4, false, 1>(P, gptrs, st);
    if (P.R == 2) return launch<GBF, 2, 2, false, 2>(P, gptrs, st);
    if (P.R <= 4) return launch<GBF, 4, 1, false, 4>(P, gptrs, st);
    if (P.R <= 32) return launch<GBF, 4, 1, true, 32>(P, gptrs, st);
    if (P.R <= 1024) return launch<GBF, 4, 1, true, 1024>(P, gptrs, st);
    return WS_ERR_TOO_LARGE;
}

}  // namespace

ws_status launch_af(const AfLaunch& P, bool gbf, const void* const* gptrs, void* clear, size_t clear_bytes, cudaStream_t st) {
    const ws_status s = launch_clear(clear, clear_bytes, P.status, st);
    if (s != WS_OK) return s;
    return gbf ? launch_r<true>(P, gptrs, st) : launch_r<false>(P, gptrs, st);
}

}  // namespace wsk
