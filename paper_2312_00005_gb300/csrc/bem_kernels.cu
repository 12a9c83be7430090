// bem_kernels.cu -- CUDA kernels (sm_103a) of the BEM + FMM matrix-vector
// product, the incident field, the field evaluation and the device-resident
// GMRES primitives.  Method: arXiv 2312.00005 (NumCalc); each kernel names
// the section or equation it computes.
#include "bem_kernels.cuh"

#include <type_traits>

namespace bem {

// ------------------------------------------------------------------ warp helpers
__device__ __forceinline__ float2 warp_sum(float2 v)
{
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// A sum of complex FP32 terms with its rounding errors beside it (two-sum), good
// to about 2^-45: the sums of a row's partial sums, whose FP64 additions cost 9 us
// of the 276 of a recomputed product on 5120 elements (a plain FP32 sum of 20
// parts loses a tenth of the product's accuracy instead).
struct Sum2 {
    float2 s, e;
    __device__ __forceinline__ Sum2() : s(make_float2(0.f, 0.f)), e(make_float2(0.f, 0.f)) {}
    __device__ __forceinline__ explicit Sum2(double2 v) : s(make_float2((float)v.x, (float)v.y))
    {
        e = make_float2((float)(v.x - (double)s.x), (float)(v.y - (double)s.y));
    }
    static __device__ __forceinline__ void add1(float &s, float &e, float a)
    {
        const float t = __fadd_rn(s, a), b = __fsub_rn(t, s);
        e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(a, b)));
        s = t;
    }
    __device__ __forceinline__ void add(float2 a)
    {
        add1(s.x, e.x, a.x);
        add1(s.y, e.y, a.y);
    }
    __device__ __forceinline__ float2 value() const { return make_float2(s.x + e.x, s.y + e.y); }
    __device__ __forceinline__ double2 value_d() const
    {
        return make_double2((double)s.x + (double)e.x, (double)s.y + (double)e.y);
    }
};
// the sum over the lanes that differ by multiples of w (a power of two)
__device__ __forceinline__ float2 lanes_sum(float2 v, int w)
{
    for (int o = w; o < 32; o <<= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// ------------------------------------------------------------------ near field
// Expensive pairs (heavy_rt2) of the stored near field, listed by kind so
// that the warps of k_near_store_heavy take pairs of one kind: 0 = self term,
// 1 = subdivided element, 1 + m = regular order m >= 4 (a sorting hint from
// FP32 r~; the heavy kernel decides the rules itself).  Pass 1 (heavy null)
// counts per kind; pass 2 writes each pair at off[kind] + its rank.
__global__ void k_near_classify(NearArgs a, int2 *__restrict__ heavy, unsigned long long *count,
                                const unsigned long long *off)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= a.E.n) return;
    const QuadTables &Q = *a.Q;
    const float3 xhi = f3(a.E.chi[i]), xlo = f3(a.E.clo[i]);
    const int t = a.N.leaf_of[i];
    const int r_end = a.N.run_ptr[t + 1], nc = a.N.ncol[t];
    int r = a.N.run_ptr[t];
    for (int p = lane; p < nc; p += 32) {
        const int j = near_col(a.N, r_end, r, p);
        const float4 cj = a.E.chi[j];
        float3 D0;
        const float rt2 = pair_rt2(f3(cj), f3(a.E.clo[j]), xhi, xlo, __frcp_rn(cj.w), D0);
        if (!heavy_rt2(i, j, rt2, Q)) continue;
        int kind;
        if (i == j) {
            kind = 0;
        } else if (rt2 < Q.rt_sub * Q.rt_sub) {
            kind = 1;
        } else {
            int m = 1;
            while (m < Q.m_max && !(rt2 > Q.R2[m])) ++m;
            kind = 1 + m;
        }
        const unsigned long long q = atomicAdd(count + kind, 1ull);
        if (heavy) heavy[off[kind] + q] = make_int2((int)i, p);
    }
}

// Near-field entries except the expensive pairs (self, order >= 4 or
// subdivided: k_near_store_heavy).  One block per (leaf, 256 columns): a
// thread holds its column's element data in registers and walks the leaf's
// rows, whose data sit in shared memory (broadcast reads); the 32 columns of
// a warp then write 32 consecutive values of one row.  r~ is compared in
// squared form (FP64 when within 2e-5 of a threshold).  Four blocks per SM
// (64 registers, a few spilled) keep more warps issuing than two blocks
// with every value in registers.  (Orders 2 and 3 in place instead of queued, as
// in the recomputed product: 633 us against 502 on 20,480 elements, since only
// two thirds of a warp's lanes agree on the order.)
constexpr int kLightRows = 64;
// the general rule out of line, so that the common path keeps few registers
__device__ __noinline__ bool general_entry(const NearArgs &a, int64_t i, int64_t j, float2 *out)
{
    const double xd[3] = {a.E.cd[3 * i], a.E.cd[3 * i + 1], a.E.cd[3 * i + 2]};
    return bm_entry(a.E, i, j, f3(a.E.chi[i]), f3(a.E.clo[i]), xd, f3(a.E.nrm[i]), a.k, a.ik_inv, a.tau, *a.Q, a.cp[j],
                    a.cq[j], *out);
}
// Entry A_ij of order 2 or 3 over the whole element j (no subdivision).
__device__ __forceinline__ float2 order23_entry(const ElemDev &E, int j, float3 D0, float3 nx, float k, float ik_inv,
                                                const QuadTables &Q, int code, float2 cpj, float2 cqj)
{
    const float4 cj = E.chi[j];
    const float3 ny = f3(E.nrm[j]), e1 = f3(E.e1[j]), e2 = f3(E.e2[j]);
    const float3 base = add3(D0, f3(E.va[j]));          // a - x
    float2 Kp = make_float2(0.f, 0.f), Kq = Kp;
    const int nq = code * code;
    for (int u = 0; u < nq; ++u) {
        const float3 d = mad3(Q.tri_eta[code][u], e2, mad3(Q.tri_xi[code][u], e1, base));
        bm_point(d, nx, ny, k, ik_inv, 2.0f * cj.w * Q.tri_w[code][u], Kp, Kq);
    }
    return cadd(cmul(cpj, Kp), cmul(cqj, Kq));
}

__global__ void __launch_bounds__(256, 4) k_near_store_light(NearArgs a, float2 *__restrict__ val,
                                                          int *__restrict__ err)
{
    __shared__ float4 s_hi[kLightRows], s_lo[kLightRows], s_n[kLightRows];
    __shared__ double s_xd[kLightRows][3];
    __shared__ int64_t s_rp[kLightRows];
    // per warp: queued order-2 / order-3 entries (row slot, column position, column)
    __shared__ int3 s_q[8][2][64];
    const int t = blockIdx.x;
    const int nc = a.N.ncol[t];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = blockIdx.y * blockDim.x + threadIdx.x;
    if ((int)(blockIdx.y * blockDim.x) >= nc) return;
    const QuadTables &Q = *a.Q;
    const int64_t e0 = a.N.leaf_start[t], e1 = a.N.leaf_start[t + 1];
    const bool live = p < nc;
    const unsigned lt = (1u << lane) - 1u;
    // this thread's column: binary search of the leaf's runs
    int j = 0;
    float4 cj = make_float4(0.f, 0.f, 0.f, 1.f), lj = cj, nj = cj;
    float2 cpj = make_float2(0.f, 0.f), cqj = cpj;
    if (live) {
        int lo = a.N.run_ptr[t], hi = a.N.run_ptr[t + 1] - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.N.runs[mid].y <= p) lo = mid;
            else hi = mid - 1;
        }
        const int2 rr = a.N.runs[lo];
        j = rr.x + (p - rr.y);
        cj = a.E.chi[j];
        lj = a.E.clo[j];
        nj = a.E.nrm[j];
        cpj = a.cp[j];
        cqj = a.cq[j];
    }
    const float inv_area = __frcp_rn(cj.w);
    int nq2 = 0, nq3 = 0;      // warp-uniform queue lengths
    // computes 32 queued entries of order c (one per lane; fewer on a flush)
    auto run_queue = [&](int c, int cnt) {
        if (lane < cnt) {
            const int3 e = s_q[warp][c - 2][lane];
            const float4 cjq = a.E.chi[e.z];
            float3 D0;
            pair_rt2(f3(cjq), f3(a.E.clo[e.z]), f3(s_hi[e.x]), f3(s_lo[e.x]), __frcp_rn(cjq.w), D0);
            val[s_rp[e.x] + e.y] = order23_entry(a.E, e.z, D0, f3(s_n[e.x]), a.k, a.ik_inv, Q, c, a.cp[e.z], a.cq[e.z]);
        }
        __syncwarp();
        // keep the entries beyond the first 32
        const int rest = cnt > 32 ? cnt - 32 : 0;
        int3 keep = make_int3(0, 0, 0);
        if (lane < rest) keep = s_q[warp][c - 2][32 + lane];
        __syncwarp();
        if (lane < rest) s_q[warp][c - 2][lane] = keep;
        __syncwarp();
        return rest;
    };
    for (int64_t b0 = e0; b0 < e1; b0 += kLightRows) {
        const int nr = (int)min((int64_t)kLightRows, e1 - b0);
        __syncthreads();
        for (int q = threadIdx.x; q < nr; q += blockDim.x) {
            s_hi[q] = a.E.chi[b0 + q];
            s_lo[q] = a.E.clo[b0 + q];
            s_n[q] = a.E.nrm[b0 + q];
            s_xd[q][0] = a.E.cd[3 * (b0 + q)];
            s_xd[q][1] = a.E.cd[3 * (b0 + q) + 1];
            s_xd[q][2] = a.E.cd[3 * (b0 + q) + 2];
            s_rp[q] = a.N.row_ptr[b0 + q];
        }
        __syncthreads();
        for (int q = 0; q < nr; ++q) {
            const int64_t i = b0 + q;
            int code = -1;
            float3 D0 = make_float3(0.f, 0.f, 0.f);
            if (live) {
                const float3 xhi = f3(s_hi[q]), xlo = f3(s_lo[q]);
                const float rt2 = pair_rt2(f3(cj), f3(lj), xhi, xlo, inv_area, D0);
                if (!heavy_rt2(i, j, rt2, Q)) {
                    if (Q.m_max > 3) {
                        const float g = 2e-5f;
                        if (fabsf(rt2 - Q.R2[1]) <= g * Q.R2[1] || fabsf(rt2 - Q.R2[2]) <= g * Q.R2[2]) {
                            double d[3];
                            for (int c = 0; c < 3; ++c)
                                d[c] = (s_xd[q][c] - a.E.cd[3 * j + c]) -
                                       (a.E.vad[3 * j + c] + (1.0 / 3.0) * a.E.e1d[3 * j + c] +
                                        (1.0 / 3.0) * a.E.e2d[3 * j + c]);
                            code = rule_from_rt_d(sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) / sqrt(a.E.ad[j]), Q);
                        } else {
                            code = rt2 > Q.R2[1] ? 1 : (rt2 > Q.R2[2] ? 2 : 3);
                        }
                    } else {
                        code = 0;
                    }
                }
            }
            if (code == 1) {
                // the 1 x 1 conical rule is the centroid rule
                float2 Kp = make_float2(0.f, 0.f), Kq = Kp;
                bm_point(D0, f3(s_n[q]), f3(nj), a.k, a.ik_inv, cj.w, Kp, Kq);
                val[s_rp[q] + p] = cadd(cmul(cpj, Kp), cmul(cqj, Kq));
            } else if (code == 0) {
                // subdivision or a high order (only when the heavy split is
                // off, m_max <= 3): the general rule
                float2 v;
                if (!general_entry(a, i, j, &v)) {
                    atomicMin(err, j);
                    v = make_float2(0.f, 0.f);
                }
                val[s_rp[q] + p] = v;
            }
            // queue orders 2 and 3 for batches of one order
            const unsigned m2 = __ballot_sync(0xffffffffu, code == 2), m3 = __ballot_sync(0xffffffffu, code == 3);
            if (code == 2) s_q[warp][0][nq2 + __popc(m2 & lt)] = make_int3(q, p, j);
            if (code == 3) s_q[warp][1][nq3 + __popc(m3 & lt)] = make_int3(q, p, j);
            nq2 += __popc(m2);
            nq3 += __popc(m3);
            __syncwarp();
            if (nq2 >= 32) nq2 = run_queue(2, nq2);
            if (nq3 >= 32) nq3 = run_queue(3, nq3);
        }
        // the rows' data are replaced next: flush
        while (nq2 > 0) nq2 = run_queue(2, nq2);
        while (nq3 > 0) nq3 = run_queue(3, nq3);
    }
}

// Stored near field, expensive pairs: one thread per listed pair.
__global__ void k_near_store_heavy(NearArgs a, const int2 *__restrict__ heavy, int64_t nheavy,
                                   float2 *__restrict__ val, int *__restrict__ err)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nheavy) return;
    const int2 ip = heavy[q];
    const int64_t i = ip.x;
    const QuadTables &Q = *a.Q;
    const float4 ch = a.E.chi[i], cl = a.E.clo[i];
    const float3 xhi = f3(ch), xlo = f3(cl), nx = f3(a.E.nrm[i]);
    const double xd[3] = {a.E.cd[3 * i], a.E.cd[3 * i + 1], a.E.cd[3 * i + 2]};
    const int t = a.N.leaf_of[i];
    int r = a.N.run_ptr[t];
    const int j = near_col(a.N, a.N.run_ptr[t + 1], r, ip.y);
    float2 v;
    if (!bm_entry(a.E, i, j, xhi, xlo, xd, nx, a.k, a.ik_inv, a.tau, Q, a.cp[j], a.cq[j], v)) {
        atomicMin(err, j);
        v = make_float2(0.f, 0.f);
    }
    val[a.N.row_ptr[i] + ip.y] = v;
}

// Near-field product with stored entries: y_i = sum_p val[row_i + p] x[col(p)],
// one warp per row; four independent loads in flight per lane.
__global__ void k_near_spmv(NearArgs a, const float2 *__restrict__ val, const float2 *__restrict__ x,
                            float2 *__restrict__ y, const int *skip)
{
    if (skip_now(skip)) return;
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= a.E.n) return;
    const int t = a.N.leaf_of[i];
    const int r_end = a.N.run_ptr[t + 1], nc = a.N.ncol[t];
    int r = a.N.run_ptr[t];
    const float2 *__restrict__ v = val + a.N.row_ptr[i];
    float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
    int p = lane;
    for (; p + 96 < nc; p += 128) {
        const float2 v0 = __ldcs(v + p), v1 = __ldcs(v + p + 32), v2 = __ldcs(v + p + 64), v3 = __ldcs(v + p + 96);
        const int j0 = near_col(a.N, r_end, r, p);
        const int j1 = near_col(a.N, r_end, r, p + 32);
        const int j2 = near_col(a.N, r_end, r, p + 64);
        const int j3 = near_col(a.N, r_end, r, p + 96);
        acc0 = cfma(v0, x[j0], acc0);
        acc1 = cfma(v1, x[j1], acc1);
        acc0 = cfma(v2, x[j2], acc0);
        acc1 = cfma(v3, x[j3], acc1);
    }
    for (; p < nc; p += 32) acc0 = cfma(__ldcs(v + p), x[near_col(a.N, r_end, r, p)], acc0);
    float2 acc = warp_sum(cadd(acc0, acc1));
    if (lane == 0) y[i] = acc;
}

// Stored near field (Sec. 3.3.3, matrix N) over work items: an item is a
// range of rows of one leaf; the leaf's near columns x are staged in shared
// memory (kept while consecutive items share the leaf) and the item's values
// (rows x ncol, contiguous) are split evenly among the warps, which stream
// them from HBM (evict-first, 8 loads per lane in flight: enough for
// the bandwidth with 8 blocks per SM, and few registers, which the far-field
// kernels running beside need).  Each warp
// leaves a partial per row it touched; the block sums them in warp order.
// One block per item: items are small, so the block scheduler balances the
// work across SMs (and shares them with the far-field kernels running
// beside) whatever the leaf sizes.
// Streamed 16-byte load of stored values: read-only path, no L1 allocation,
// and an L2 fetch of the surrounding 256 bytes (the next lanes' values).
__device__ __forceinline__ float4 ld_stream4(const float4 *p)
{
    float4 v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ float2 spmv_segment(const float2 *__restrict__ v, const float2 *__restrict__ xs, int c0,
                                               int c1, int lane)
{
    // sum_{c0 <= c < c1} v[c] xs[c] with c0 even: column pairs per 16-byte
    // load (v and xs 16-byte aligned), the odd last column alone
    const float4 *__restrict__ v4 = reinterpret_cast<const float4 *>(v);
    const float4 *__restrict__ x4 = reinterpret_cast<const float4 *>(xs);
    float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0, acc2 = acc0, acc3 = acc0;
    int q = (c0 >> 1) + lane;
    const int qe = c1 >> 1;
    for (; q + 224 < qe; q += 256) {
        float4 vv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) vv[u] = ld_stream4(v4 + q + 32 * u);
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            const float4 xa = x4[q + 32 * u], xb = x4[q + 32 * (u + 1)];
            acc0 = cfma(make_float2(vv[u].x, vv[u].y), make_float2(xa.x, xa.y), acc0);
            acc1 = cfma(make_float2(vv[u].z, vv[u].w), make_float2(xa.z, xa.w), acc1);
            acc2 = cfma(make_float2(vv[u + 1].x, vv[u + 1].y), make_float2(xb.x, xb.y), acc2);
            acc3 = cfma(make_float2(vv[u + 1].z, vv[u + 1].w), make_float2(xb.z, xb.w), acc3);
        }
    }
    for (; q + 96 < qe; q += 128) {
        float4 vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) vv[u] = ld_stream4(v4 + q + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
            const float4 xa = x4[q + 32 * u], xb = x4[q + 32 * (u + 1)];
            acc0 = cfma(make_float2(vv[u].x, vv[u].y), make_float2(xa.x, xa.y), acc0);
            acc1 = cfma(make_float2(vv[u].z, vv[u].w), make_float2(xa.z, xa.w), acc1);
            acc2 = cfma(make_float2(vv[u + 1].x, vv[u + 1].y), make_float2(xb.x, xb.y), acc2);
            acc3 = cfma(make_float2(vv[u + 1].z, vv[u + 1].w), make_float2(xb.z, xb.w), acc3);
        }
    }
    for (; q < qe; q += 32) {
        const float4 vv = ld_stream4(v4 + q), xa = x4[q];
        acc0 = cfma(make_float2(vv.x, vv.y), make_float2(xa.x, xa.y), acc0);
        acc1 = cfma(make_float2(vv.z, vv.w), make_float2(xa.z, xa.w), acc1);
    }
    if ((c1 & 1) && lane == 0) acc2 = cfma(v[c1 - 1], xs[c1 - 1], acc2);
    return warp_sum(cadd(cadd(acc0, acc1), cadd(acc2, acc3)));
}

__global__ void __launch_bounds__(kSpmvThreads) k_near_spmv_items(NearArgs a, const int4 *__restrict__ items,
                                                                  const float2 *__restrict__ val,
                                                                  const float2 *__restrict__ x,
                                                                  float2 *__restrict__ y, const int *skip)
{
    if (skip_now(skip)) return;
    extern __shared__ float2 xs[];
    constexpr int kW = kSpmvThreads / 32;
    static_assert(kSpmvMaxItemRows * kW == kSpmvThreads, "one partial slot per thread");
    __shared__ float2 part[kSpmvMaxItemRows][kW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int4 W = items[blockIdx.x];
    const int t = W.x;
    const int nc = a.N.ncol[t];
    {
        const int r0 = a.N.run_ptr[t], r1 = a.N.run_ptr[t + 1];
        for (int r = r0 + warp; r < r1; r += kW) {
            const int2 rr = a.N.runs[r];
            const int end = (r + 1 < r1) ? a.N.runs[r + 1].y : nc;
            int p = rr.y + lane;
            for (; p + 224 < end; p += 256) {
                float2 t8[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) t8[u] = x[rr.x + (p + 32 * u - rr.y)];
#pragma unroll
                for (int u = 0; u < 8; ++u) xs[p + 32 * u] = t8[u];
            }
            for (; p < end; p += 32) xs[p] = x[rr.x + (p - rr.y)];
        }
    }
    part[threadIdx.x / kW][threadIdx.x % kW] = make_float2(0.f, 0.f);
    __syncthreads();
    const int64_t i0 = a.N.leaf_start[t] + W.y;
    const int nrow = min(W.z - W.y, kSpmvMaxItemRows);   // the host never makes larger items
    // the item's rows (stride ncp, padded to even) split at even positions
    const int ncp = (nc + 1) & ~1;
    const int64_t total = (int64_t)nrow * ncp;
    int64_t qa = (total * warp / kW) & ~(int64_t)1;
    const int64_t qb = warp == kW - 1 ? total : (total * (warp + 1) / kW) & ~(int64_t)1;
    while (qa < qb) {
        const int r = (int)(qa / ncp);
        const int c0 = (int)(qa - (int64_t)r * ncp);
        const int c1 = (int)min((int64_t)ncp, (int64_t)c0 + (qb - qa));
        const int c1r = min(c1, nc);
        if (c0 < c1r) {
            const float2 acc = spmv_segment(val + a.N.row_ptr[i0 + r], xs, c0, c1r, lane);
            if (lane == 0) part[r][warp] = acc;
        }
        qa += c1 - c0;
    }
    __syncthreads();
    if (threadIdx.x < nrow) {
        float2 sum = part[threadIdx.x][0];
#pragma unroll
        for (int w = 1; w < kW; ++w) sum = cadd(sum, part[threadIdx.x][w]);
        y[i0 + threadIdx.x] = sum;
    }
}

// A^T from the stored values of A, in A's layout: the rows j of leaf t, each
// padded to an even length ncp (the stride of t's rows), take at column c
// the value A_i,j of t's c-th transposed row i, which sits at trow_off[k0 +
// c] + (j - t0).  Threads take consecutive columns of a row (coalesced
// writes); the reads are the scattered column segments.
__global__ void k_near_transpose(const int64_t *__restrict__ leaf_start, const int *__restrict__ trow_ptr,
                                 const int64_t *__restrict__ trow_off, const int64_t *__restrict__ row_ptr,
                                 const float2 *__restrict__ val, float2 *__restrict__ valT)
{
    const int t = blockIdx.x;
    const int64_t t0 = leaf_start[t];
    const int nt = (int)(leaf_start[t + 1] - t0);
    const int k0 = trow_ptr[t], nk = trow_ptr[t + 1] - k0;
    const int ncp = (nk + 1) & ~1;
    const int64_t total = (int64_t)nt * ncp;
    for (int64_t idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int jj = (int)(idx / ncp), c = (int)(idx - (int64_t)jj * ncp);
        valT[row_ptr[t0 + jj] + c] = c < nk ? val[trow_off[k0 + c] + jj] : make_float2(0.f, 0.f);
    }
}

// Transposed near-field product from the stored values (the near relation
// of the leaves being symmetric): for the elements j of leaf t = blockIdx.x,
//   y_j = sum_{s in near(t)} sum_{i in s} A_ij x_i,
// where A_ij sits at trow_off[k] + (j - first element of t) for row k of the
// leaf's list.  A warp takes R = 32 / w rows at a time (w the power of two at
// or above the leaf size, at most 32): lane (sub, jj) reads one row's value at
// column jj of a w-wide segment (a coalesced run per row); the sub-rows' and
// then the warps' sums are added in a fixed order.
__global__ void __launch_bounds__(kSpmvTThreads) k_near_spmv_t(const int64_t *__restrict__ leaf_start,
                                                               const int *__restrict__ trow_ptr,
                                                               const int *__restrict__ trow_i,
                                                               const int64_t *__restrict__ trow_off,
                                                               const float2 *__restrict__ val,
                                                               const float2 *__restrict__ x, float2 *__restrict__ y,
                                                               const int *skip)
{
    if (skip_now(skip)) return;
    constexpr int kW = kSpmvTThreads / 32;
    __shared__ float2 part[kW][32];
    const int t = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = leaf_start[t];
    const int cnt = (int)(leaf_start[t + 1] - j0);
    int w = 1;
    while (w < cnt && w < 32) w <<= 1;
    const int R = 32 / w, sub = lane / w, jj = lane % w;
    const int k0 = trow_ptr[t], k1 = trow_ptr[t + 1];
    for (int c0 = 0; c0 < cnt; c0 += w) {
        const bool live = c0 + jj < cnt;
        float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
        int k = k0 + warp * R + sub;
        const int step = kW * R;
        // kTU rows per warp step: their positions first, then all their
        // values and x in flight together
        constexpr int kTU = 4;
        for (; k + (kTU - 1) * step < k1; k += kTU * step) {
            int iv[kTU];
            int64_t ov[kTU];
#pragma unroll
            for (int u = 0; u < kTU; ++u) {
                iv[u] = trow_i[k + u * step];
                ov[u] = trow_off[k + u * step];
            }
            float2 xv[kTU], vv[kTU];
#pragma unroll
            for (int u = 0; u < kTU; ++u) {
                xv[u] = x[iv[u]];
                vv[u] = live ? __ldcs(val + ov[u] + c0 + jj) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < kTU; u += 2) {
                acc0 = cfma(vv[u], xv[u], acc0);
                acc1 = cfma(vv[u + 1], xv[u + 1], acc1);
            }
        }
        for (; k < k1; k += step)
            if (live) acc0 = cfma(__ldcs(val + trow_off[k] + c0 + jj), x[trow_i[k]], acc0);
        float2 acc = cadd(acc0, acc1);
        // add the R sub-rows (lanes jj, jj + w, ...) in a fixed order
        for (int o = w; o < 32; o <<= 1) {
            acc.x += __shfl_down_sync(0xffffffffu, acc.x, o);
            acc.y += __shfl_down_sync(0xffffffffu, acc.y, o);
        }
        if (sub == 0) part[warp][jj] = acc;
        __syncthreads();
        if (warp == 0 && lane < w && c0 + lane < cnt) {
            float2 sum = part[0][lane];
#pragma unroll
            for (int v = 1; v < kW; ++v) sum = cadd(sum, part[v][lane]);
            y[j0 + c0 + lane] = sum;
        }
        __syncthreads();
    }
}

// sum_{c0 <= c < c1} v[c] xs_r[c] for the planes r < nr of xs (ncp floats2
// apart), as spmv_segment for one plane: each 16-byte load of v serves all
// planes.
__device__ __forceinline__ void spmv_segment_multi(const float2 *__restrict__ v, const float2 *__restrict__ xs, int ncp,
                                                   int c0, int c1, int lane, int nr, float2 out[kMaxPlanes])
{
    const float4 *__restrict__ v4 = reinterpret_cast<const float4 *>(v);
    float2 acc0[kMaxPlanes], acc1[kMaxPlanes];
#pragma unroll
    for (int r = 0; r < kMaxPlanes; ++r) acc0[r] = acc1[r] = make_float2(0.f, 0.f);
    int q = (c0 >> 1) + lane;
    const int qe = c1 >> 1;
    for (; q + 96 < qe; q += 128) {
        float4 vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) vv[u] = ld_stream4(v4 + q + 32 * u);
#pragma unroll
        for (int r = 0; r < kMaxPlanes; ++r) {
            if (r >= nr) break;
            const float4 *__restrict__ x4 = reinterpret_cast<const float4 *>(xs + (int64_t)r * ncp);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 xa = x4[q + 32 * u];
                acc0[r] = cfma(make_float2(vv[u].x, vv[u].y), make_float2(xa.x, xa.y), acc0[r]);
                acc1[r] = cfma(make_float2(vv[u].z, vv[u].w), make_float2(xa.z, xa.w), acc1[r]);
            }
        }
    }
    for (; q < qe; q += 32) {
        const float4 vv = ld_stream4(v4 + q);
#pragma unroll
        for (int r = 0; r < kMaxPlanes; ++r) {
            if (r >= nr) break;
            const float4 xa = reinterpret_cast<const float4 *>(xs + (int64_t)r * ncp)[q];
            acc0[r] = cfma(make_float2(vv.x, vv.y), make_float2(xa.x, xa.y), acc0[r]);
            acc1[r] = cfma(make_float2(vv.z, vv.w), make_float2(xa.z, xa.w), acc1[r]);
        }
    }
    if ((c1 & 1) && lane == 0) {
        const float2 vl = v[c1 - 1];
#pragma unroll
        for (int r = 0; r < kMaxPlanes; ++r)
            if (r < nr) acc0[r] = cfma(vl, xs[(int64_t)r * ncp + c1 - 1], acc0[r]);
    }
#pragma unroll
    for (int r = 0; r < kMaxPlanes; ++r) out[r] = warp_sum(cadd(acc0[r], acc1[r]));
}

template <int kThreads>
__device__ __forceinline__ void spmv_items_multi_body(const NearArgs &a, const int4 *__restrict__ items,
                                                      const float2 *__restrict__ val, const float2 *__restrict__ x,
                                                      float2 *__restrict__ y, int nr, int64_t plane, int cw)
{
    extern __shared__ float2 xs[];            // [nr][cw]: one chunk of the leaf's columns
    constexpr int kW = kThreads / 32;
    __shared__ float2 part[kMaxPlanes][kSpmvMaxItemRows][kW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int4 W = items[blockIdx.x];
    const int t = W.x;
    const int nc = a.N.ncol[t];
    const int ncp = (nc + 1) & ~1;
    const int run0 = a.N.run_ptr[t], run1 = a.N.run_ptr[t + 1];
    for (int q = threadIdx.x; q < kMaxPlanes * kSpmvMaxItemRows * kW; q += kThreads)
        (&part[0][0][0])[q] = make_float2(0.f, 0.f);
    const int64_t i0 = a.N.leaf_start[t] + W.y;
    const int nrow = min(W.z - W.y, kSpmvMaxItemRows);
    // the columns in chunks of cw (even, so every chunk's rows start on a
    // 16-byte boundary); each warp keeps its partial sums of a row in its
    // own slot of part across the chunks
    for (int cb = 0; cb < ncp; cb += cw) {
        const int cwp = min(cw, ncp - cb);
        const int ce = min(cb + cwp, nc);
        if (cb > 0) __syncthreads();          // the previous chunk's columns are no longer read
        for (int r = run0 + warp; r < run1; r += kW) {
            const int2 rr = a.N.runs[r];
            const int end = (r + 1 < run1) ? a.N.runs[r + 1].y : nc;
            const int lo = max(rr.y, cb), hi = min(end, ce);
            for (int p = lo + lane; p < hi; p += 32)
                for (int pl = 0; pl < nr; ++pl) xs[pl * cw + (p - cb)] = x[pl * plane + rr.x + (p - rr.y)];
        }
        __syncthreads();
        const int64_t total = (int64_t)nrow * cwp;
        int64_t qa = (total * warp / kW) & ~(int64_t)1;
        const int64_t qb = warp == kW - 1 ? total : (total * (warp + 1) / kW) & ~(int64_t)1;
        while (qa < qb) {
            const int r = (int)(qa / cwp);
            const int c0 = (int)(qa - (int64_t)r * cwp);
            const int c1 = (int)min((int64_t)cwp, (int64_t)c0 + (qb - qa));
            const int c1r = min(c1, ce - cb);
            if (c0 < c1r) {
                float2 acc[kMaxPlanes];
                spmv_segment_multi(val + a.N.row_ptr[i0 + r] + cb, xs, cw, c0, c1r, lane, nr, acc);
                if (lane == 0)
#pragma unroll
                    for (int pl = 0; pl < kMaxPlanes; ++pl) part[pl][r][warp] = cadd(part[pl][r][warp], acc[pl]);
            }
            qa += c1 - c0;
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < nrow * nr; q += kThreads) {
        const int row = q % nrow, pl = q / nrow;
        float2 sum = part[pl][row][0];
#pragma unroll
        for (int w = 1; w < kW; ++w) sum = cadd(sum, part[pl][row][w]);
        y[pl * plane + i0 + row] = sum;
    }
}

#define BEM_SPMV_MULTI_KERNEL(NAME, THREADS)                                                                          \
    __global__ void __launch_bounds__(THREADS)                                                                       \
        NAME(NearArgs a, const int4 *__restrict__ items, const float2 *__restrict__ val, const float2 *__restrict__ x, \
             float2 *__restrict__ y, int nr, int64_t plane, int cw, const int *skip)                                 \
    {                                                                                                                 \
        if (skip_now(skip)) return;                                                                                   \
        spmv_items_multi_body<THREADS>(a, items, val, x, y, nr, plane, cw);                                           \
    }
BEM_SPMV_MULTI_KERNEL(k_near_spmv_items_multi, kSpmvMultiThreads)
BEM_SPMV_MULTI_KERNEL(k_near_spmv_items_multi_s, kChunkThreads)
#undef BEM_SPMV_MULTI_KERNEL

// ------------------------------------------------------------------ recomputed near field
// Kp and / or Kq of bm_point at one quadrature point (needp, needq uniform
// over the warp: a sound-hard problem has no q-columns, the admittance
// derivative's operator no p-columns).
__device__ __forceinline__ void bm_point_sel(float3 d, float3 nx, float3 ny, float k, float ik_inv, float w, bool needp,
                                             bool needq, float2 &Kp, float2 &Kq)
{
    const float r2 = dot3f(d, d);
    const float ir = rsqrtf(r2);
    const float r = r2 * ir;
    float s, c;
    sincos_turns(k * r * 0.15915494309189535f, &s, &c);
    const float g = w * ir * kInv4Pi;
    const float2 G = make_float2(c * g, s * g);
    const float rx = dot3f(d, nx) * ir;
    if (needp) {
        const float ry = dot3f(d, ny) * ir, nn = dot3f(nx, ny);
        const float ir2k = ir * ir * ik_inv;
        const float rxry = rx * ry;
        const float2 P = make_float2(ir * (ry - 3.0f * rxry + nn), -k * ry + (k - 3.0f * ir2k) * rxry + ir2k * nn);
        Kp = cfma(G, P, Kp);
    }
    if (needq) Kq = cfma(G, make_float2(1.0f - rx, -(ir * ik_inv) * rx), Kq);
}

// A part of a subdivided element, packed: the order in bits 24..26, the depth
// in 20..23 and the children taken from the whole element down, two bits
// each, in 0..19 (the first in bits 0, 1).
constexpr int kPartDepth = 10;
__device__ __forceinline__ SubTri child_triangle(const SubTri &s, unsigned i)
{
    const float mx01 = 0.5f * (s.x0 + s.x1), my01 = 0.5f * (s.y0 + s.y1);
    const float mx12 = 0.5f * (s.x1 + s.x2), my12 = 0.5f * (s.y1 + s.y2);
    const float mx20 = 0.5f * (s.x2 + s.x0), my20 = 0.5f * (s.y2 + s.y0);
    switch (i) {
        case 0: return SubTri{s.x0, s.y0, mx01, my01, mx20, my20, s.depth + 1};
        case 1: return SubTri{mx01, my01, s.x1, s.y1, mx12, my12, s.depth + 1};
        case 2: return SubTri{mx20, my20, mx12, my12, s.x2, s.y2, s.depth + 1};
        default: return SubTri{mx01, my01, mx12, my12, mx20, my20, s.depth + 1};
    }
}
// The triangle whose child i is s: exact, as the coordinates are multiples of
// 2^-kPartDepth.
__device__ __forceinline__ SubTri parent_triangle(const SubTri &s, unsigned i)
{
    switch (i) {
        case 0:
            return SubTri{s.x0, s.y0, 2.f * s.x1 - s.x0, 2.f * s.y1 - s.y0, 2.f * s.x2 - s.x0, 2.f * s.y2 - s.y0,
                          s.depth - 1};
        case 1:
            return SubTri{2.f * s.x0 - s.x1, 2.f * s.y0 - s.y1, s.x1, s.y1, 2.f * s.x2 - s.x1, 2.f * s.y2 - s.y1,
                          s.depth - 1};
        case 2:
            return SubTri{2.f * s.x0 - s.x2, 2.f * s.y0 - s.y2, 2.f * s.x1 - s.x2, 2.f * s.y1 - s.y2, s.x2, s.y2,
                          s.depth - 1};
        default:
            return SubTri{s.x0 + s.x2 - s.x1, s.y0 + s.y2 - s.y1, s.x0 + s.x1 - s.x2, s.y0 + s.y1 - s.y2,
                          s.x1 + s.x2 - s.x0, s.y1 + s.y2 - s.y0, s.depth - 1};
    }
}
__device__ __forceinline__ SubTri part_triangle(unsigned code, int depth)
{
    SubTri s{0.f, 0.f, 1.f, 0.f, 0.f, 1.f, 0};
    for (int d = 0; d < depth; ++d) s = child_triangle(s, (code >> (2 * d)) & 3u);
    return s;
}
// The parts under one rule of element j seen from x (D0 = x_j - x, xd the FP64
// point; Sec. 3.1.3's subdivision, the decisions of integrate_regular_acc),
// without integrating: their number, and the first cap codes in out.  0 when the element is subdivided deeper than a
// code can say (the caller then takes the general rule, which also reports the
// limit).
__device__ __forceinline__ int cut_element(const ElemDev &E, const QuadTables &Q, int64_t j, float3 D0, const double *xd,
                                           unsigned *out, int cap)
{
    const float area = E.chi[j].w;
    const float3 e1 = f3(E.e1[j]), e2 = f3(E.e2[j]);
    const float3 base = add3(D0, f3(E.va[j]));
    int m = whole_rule(E, j, D0, area, xd, Q);
    if (m > 0) {
        if (cap > 0) *out = (unsigned)m << 24;
        return 1;
    }
    // depth first through the children; up: the parent of the part at hand
    SubTri up{0.f, 0.f, 1.f, 0.f, 0.f, 1.f, 0};
    int n = 0;
    unsigned path = 0;                     // child path[d] taken at depth d ...
    if (Q.max_depth < 1) return 0;
    for (;;) {
        const int depth = up.depth + 1;
        const SubTri s = child_triangle(up, (path >> (2 * up.depth)) & 3u);
        const float cx = (s.x0 + s.x1 + s.x2) * (1.0f / 3.0f), cy = (s.y0 + s.y1 + s.y2) * (1.0f / 3.0f);
        m = sub_rule(E, j, mad3(cy, e2, mad3(cx, e1, base)), area * exp2f(-2.0f * (float)depth), s, xd, Q);
        if (m == 0) {
            if (depth >= kPartDepth || depth >= Q.max_depth) return 0;
            up = s;                        // down to its first child
            continue;
        }
        if (n < cap) out[n] = (unsigned)m << 24 | (unsigned)depth << 20 | path;
        ++n;
        // the next sibling, or the next one of the nearest ancestor that has one
        while (((path >> (2 * up.depth)) & 3u) == 3u) {
            path &= ~(3u << (2 * up.depth));
            if (up.depth == 0) return n;
            up = parent_triangle(up, (path >> (2 * (up.depth - 1))) & 3u);
        }
        path += 1u << (2 * up.depth);
    }
}
// The same of the pair of elements (i, j).
__device__ __noinline__ int cut_pair(const NearArgs &a, int64_t i, int64_t j, unsigned *out, int cap)
{
    const double xd[3] = {a.E.cd[3 * i], a.E.cd[3 * i + 1], a.E.cd[3 * i + 2]};
    const float3 D0 = add3(sub3f(f3(a.E.chi[j]), f3(a.E.chi[i])), sub3f(f3(a.E.clo[j]), f3(a.E.clo[i])));
    return cut_element(a.E, *a.Q, j, D0, xd, out, cap);
}

// first point of order m in a table of orders 1 to 6: 0, 1, 5, 14, 30, 55
__device__ __forceinline__ int rule_at(int m) { return (m - 1) * m * (2 * m - 1) / 6; }
// (xi, eta, 2 w) of point v of the orders 1 to 6 in a row
__device__ __forceinline__ float4 rule_point(const QuadTables &Q, int v)
{
    int m = 1;
    while (rule_at(m + 1) <= v) ++m;
    const int u = v - rule_at(m);
    return make_float4(Q.tri_xi[m][u], Q.tri_eta[m][u], 2.0f * Q.tri_w[m][u], 0.f);
}
constexpr int kCutKept = 96;                             // codes of a pair that its thread keeps (else cut again)
constexpr int kPartBytes = kFusedParts * 10;           // the parts of a block's queued pairs, in shared memory
// A block's nq queued pairs, kThreads (its threads) at a time: cut into parts
// (cut(pair, out, cap): their number, and the first cap codes), the parts sorted
// by order, integrated part by part (part(pair, code)); pairs whose parts
// found no room go into another round, pairs that cannot be cut are taken whole
// (whole(pair)).  Called by the whole block; buf: 10 kParts bytes of shared
// memory, pn: 8 counters.
template <int kThreads, int kParts, class Cut, class Part, class Whole>
__device__ __forceinline__ void work_queue(int nq, unsigned char *buf, int *pn, Cut cut, Part part, Whole whole)
{
    int *pq = reinterpret_cast<int *>(buf);                        // part: its pair
    unsigned *pc = reinterpret_cast<unsigned *>(pq + kParts); // ... its code
    unsigned short *po = reinterpret_cast<unsigned short *>(pc + kParts);   // parts by order
    int q = threadIdx.x, np = -1;                      // this thread's next pair and its parts (-1: not counted)
    unsigned codes[kCutKept];
    while (__syncthreads_or(q < nq)) {
        if (threadIdx.x < 8) pn[threadIdx.x] = 0;
        __syncthreads();
        if (q < nq) {
            if (np < 0) np = cut(q, codes, kCutKept);
            if (np > 0 && np <= kParts) {
                const int at = atomicAdd(&pn[0], np);
                if (at + np <= kParts) {
                    if (np > kCutKept) cut(q, pc + at, np);
                    for (int u = at; u < at + np; ++u) {
                        if (np <= kCutKept) pc[u] = codes[u - at];
                        pq[u] = q;
                        atomicAdd(&pn[(pc[u] >> 24) & 7], 1);
                    }
                    q += kThreads;
                    np = -1;
                } else {
                    for (int u = at; u < min(at + np, kParts); ++u) pc[u] = 0;   // order 0: no part
                }
            } else {
                whole(q);
                q += kThreads;
                np = -1;
            }
        }
        __syncthreads();
        const int n_all = min(pn[0], kParts);
        int start[8];                                  // first slot of an order: the longest first
        start[7] = 0;
        start[6] = 0;
#pragma unroll
        for (int m = 5; m >= 1; --m) start[m] = start[m + 1] + pn[m + 1];
        const int n_parts = start[1] + pn[1];
        __syncthreads();
        if (threadIdx.x < 8) pn[threadIdx.x] = 0;
        __syncthreads();
        for (int u = threadIdx.x; u < n_all; u += kThreads) {
            const int m = (pc[u] >> 24) & 7;
            if (m == 0) continue;
            int at = start[1];
#pragma unroll
            for (int v = 2; v <= 6; ++v)
                if (m == v) at = start[v];
            po[at + atomicAdd(&pn[m], 1)] = (unsigned short)u;
        }
        __syncthreads();
        for (int u = threadIdx.x; u < n_parts; u += kThreads) part(pq[po[u]], pc[po[u]]);
    }
    __syncthreads();
}

// The part's share of A_ij, to FP32 rounding; rule: (xi, eta, 2 w) of the
// points of orders 1 to 6.
__device__ __forceinline__ float2 part_entry(const NearArgs &a, int64_t i, int64_t j, unsigned code, const float4 *rule)
{
    const int m = (code >> 24) & 7, depth = (code >> 20) & 15;
    const SubTri T = part_triangle(code, depth);
    const float4 ch = a.E.chi[j];
    const float3 g1 = f3(a.E.e1[j]), g2 = f3(a.E.e2[j]), ny = f3(a.E.nrm[j]), nx = f3(a.E.nrm[i]);
    const float3 base = add3(add3(sub3f(f3(ch), f3(a.E.chi[i])), sub3f(f3(a.E.clo[j]), f3(a.E.clo[i]))), f3(a.E.va[j]));
    const float sa = ch.w * exp2f(-2.0f * (float)depth);
    const float sx1 = T.x1 - T.x0, sy1 = T.y1 - T.y0, sx2 = T.x2 - T.x0, sy2 = T.y2 - T.y0;
    float2 Kp = make_float2(0.f, 0.f), Kq = Kp;
    const int r1 = rule_at(m + 1);
    for (int v = rule_at(m); v < r1; ++v) {
        const float4 rl = rule[v];
        const float px = T.x0 + rl.x * sx1 + rl.y * sx2, py = T.y0 + rl.x * sy1 + rl.y * sy2;
        bm_point<true>(mad3(py, g2, mad3(px, g1, base)), nx, ny, a.k, a.ik_inv, sa * rl.z, Kp, Kq);
    }
    return cadd(cmul(a.cp[j], Kp), cmul(a.cq[j], Kq));
}
// v times x_w for every right-hand side, added to a row's FP64 sums (h[r][row]
// in shared memory, h at the row).
template <int NR>
__device__ __forceinline__ void add_entry(double2 *h, const float2 *__restrict__ x, int64_t n, int64_t w, float2 v)
{
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const float2 c = cmul(v, x[r * n + w]);
        atomicAdd(&h[r * kFusedRows].x, (double)c.x);
        atomicAdd(&h[r * kFusedRows].y, (double)c.y);
    }
}

// Near-field product with the entries recomputed on the fly (no storage):
// the conventional dense BEM product when the near list is everything, and
// the known boundary data's product.  Bound by FP32 / SFU issue (one kernel
// evaluation is about 55 instructions with three SFU operations), so the
// layout keeps everything else out of the inner loop and the lanes together:
//   - a lane holds one row (its midpoint and normal) in registers, the 32
//     rows being neighbours in Morton order; the columns are staged in shared
//     memory in tiles of `cols` and read as broadcasts, each warp taking an
//     eighth of a tile.  The rows of a warp see a column
//     at nearly the same distance, so they mostly agree on its rule, and no
//     sum crosses lanes until the end.  (Leaves of at most 16 rows put two
//     or more columns side by side in a warp.)
//   - orders 1 to 3 are evaluated in place; the expensive pairs (subdivided
//     elements, orders 4 to 6, distances within rounding of a threshold) are
//     queued per block and worked off after the tiles (and between two when
//     the queue is half full) by all its threads:
//     each pair is first cut into its parts under one rule (the subdivision
//     without any integration), the parts are sorted by their order, and the
//     lanes then take parts of one order, so that a warp's loops have one
//     length.  (Pairs taken whole, one per thread, had lanes of a warp in
//     different parts and orders: 7 times the instructions.)  The self terms
//     take a warp each.  The sums of all these are FP64 additions of FP32
//     terms in shared memory, exact while a row's terms lie within a factor of
//     2^20, so their order does not show; a pair that finds the queue full
//     waits for its next filling, so that every pair is taken the same way.
// A block takes the rows of one task and every gridDim.y-th part of the
// tiles; with several parts, k_near_fused_sum adds them in order.  NR right-
// hand sides share every entry.  One warp per row with lanes over the columns
// (96 bytes of element data per pair through L1, all rules mixed in a warp)
// took 721 us on 5120 elements; this takes 254 us.
// kT: the transposed product (the lists read backwards): a lane holds
// column j, the rows i whose leaves are in the near list of j's own leaf are
// staged, y_j = cp_j sum_i Kp_ij x_i + cq_j sum_i Kq_ij x_i.
template <int NR, bool kT>
__device__ __forceinline__ void near_fused_body(const NearArgs &a, const int4 *__restrict__ tasks, int rows, int cols,
                                                const float2 *__restrict__ x, float2 *__restrict__ out,
                                                int *__restrict__ err)
{
    static_assert(!kT || NR == 1, "the transposed product has one right-hand side");
    constexpr int kW = kFusedThreads / 32;
    constexpr bool kFold = !kT && NR == 1;             // the column's x folded into its coefficients
    static_assert(kFusedTile == kFusedThreads, "one staged element per thread");
    // the staged tile (a transposed product stages rows: no vertices and
    // coefficients), and afterwards the parts of the queued pairs
    constexpr int kTileArrays = kT ? 3 : 7;
    constexpr int kTileBytes = kTileArrays * kFusedTile * 16;
    __shared__ __align__(16) unsigned char s_buf[kTileBytes > kPartBytes ? kTileBytes : kPartBytes];
    float4 *s_hi = reinterpret_cast<float4 *>(s_buf), *s_lo = s_hi + kFusedTile, *s_n = s_lo + kFusedTile;
    float4 *s_va = kT ? s_hi : s_n + kFusedTile, *s_e1 = kT ? s_hi : s_va + kFusedTile;
    float4 *s_e2 = kT ? s_hi : s_e1 + kFusedTile, *s_c = kT ? s_hi : s_e2 + kFusedTile;
    __shared__ float2 s_x[NR][kFold ? 1 : kFusedTile];
    __shared__ int s_j[kFusedTile];
    __shared__ int s_qj[kFusedQueue];                  // expensive pairs: staged element and row
    __shared__ unsigned char s_qr[kFusedQueue];
    __shared__ int s_qn, s_pn[8];
    __shared__ int s_self[kFusedRows];                 // the row's own element is in this block's part
    __shared__ double2 s_h[NR][kFusedRows];
    __shared__ float4 s_rule[91];                      // (xi, eta, 2 w) of orders 1 to 6, order m from rule_at(m)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const QuadTables &Q = *a.Q;
    int t = 0;
    int64_t e0, e1;
    if (tasks) {
        const int4 T = tasks[blockIdx.x];
        t = T.x;
        e0 = T.y;
        e1 = T.z;
    } else {                                           // one leaf holds every element
        e0 = (int64_t)blockIdx.x * rows;
        e1 = min(a.E.n, e0 + rows);
    }
    const int cnt = (int)(e1 - e0);
    int w = 1;
    while (w < cnt) w <<= 1;                           // cnt <= kFusedRows = 32
    const int R = 32 / w, sub = lane / w, rr = lane % w;
    const bool live = rr < cnt;
    const int64_t e = e0 + (live ? rr : 0);
    if (threadIdx.x == 0) s_qn = 0;
    if (threadIdx.x < kFusedRows) s_self[threadIdx.x] = 0;
    if (threadIdx.x < kFusedRows)
#pragma unroll
        for (int r = 0; r < NR; ++r) s_h[r][threadIdx.x] = make_double2(0.0, 0.0);
    if (threadIdx.x < 91) s_rule[threadIdx.x] = rule_point(Q, threadIdx.x);
    // this lane's element
    const float4 ehi = a.E.chi[e], elo = a.E.clo[e], en = a.E.nrm[e];
    float3 eva = make_float3(0.f, 0.f, 0.f), ee1 = eva, ee2 = eva;
    float2 ecp = make_float2(0.f, 0.f), ecq = ecp;
    float einv = 0.f;
    bool needp = true, needq = false;
    if (kT) {
        eva = f3(a.E.va[e]);
        ee1 = f3(a.E.e1[e]);
        ee2 = f3(a.E.e2[e]);
        ecp = a.cp[e];
        ecq = a.cq[e];
        einv = __frcp_rn(ehi.w);
        needp = __any_sync(0xffffffffu, ecp.x != 0.f || ecp.y != 0.f);
        needq = __any_sync(0xffffffffu, ecq.x != 0.f || ecq.y != 0.f);
    }
    // thresholds on r~^2: order 1 clearly above R_1 and rt_sub; orders 2 and 3
    // above heavy_rt2 (m_max <= 3: rt_sub, all regular orders being among them)
    // and not within 2e-5 of R_1 or R_2 (R2[m] = 0 from m_max on: m_max = 2 has
    // no order 3 and m_max = 1 no order 2 here)
    const float rt1 = fmaxf(Q.R2[1] * (1.0f + 2e-5f), Q.whole_rt2);
    const float rt1lo = Q.R2[1] * (1.0f - 2e-5f), rt2hi = Q.R2[2] * (1.0f + 2e-5f), rt2lo = Q.R2[2] * (1.0f - 2e-5f);
    const float rth = Q.m_max > 3 ? Q.heavy_rt2 : Q.whole_rt2;
    const float k = a.k, ik_inv = a.ik_inv;
    float2 acc[NR], accq = make_float2(0.f, 0.f);      // kT: acc[0] the p sum, accq the q sum
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] = make_float2(0.f, 0.f);
    // the queued pairs (called by the whole block after a barrier; takes the
    // staged tile's place)
    auto drain = [&]() {
        auto row_of = [&](int q) { return kT ? (int64_t)s_qj[q] : e0 + s_qr[q]; };
        auto col_of = [&](int q) { return kT ? e0 + s_qr[q] : (int64_t)s_qj[q]; };
        work_queue<kFusedThreads, kFusedParts>(
            min(s_qn, kFusedQueue), s_buf, s_pn,
            [&](int q, unsigned *out, int cap) { return cut_pair(a, row_of(q), col_of(q), out, cap); },
            [&](int q, unsigned code) {
                add_entry<NR>(&s_h[0][s_qr[q]], x, a.E.n, s_qj[q], part_entry(a, row_of(q), col_of(q), code, s_rule));
            },
            [&](int q) {                               // cut deeper than a code can say
                float2 v;
                if (general_entry(a, row_of(q), col_of(q), &v)) add_entry<NR>(&s_h[0][s_qr[q]], x, a.E.n, s_qj[q], v);
                else atomicMin(err, (int)col_of(q));
            });
        if (threadIdx.x == 0) s_qn = 0;
    };
    const int nc = a.N.ncol[t];
    const int ntile = (nc + cols - 1) / cols, chunk = cols / kW;
    const int run0 = a.N.run_ptr[t], run1 = a.N.run_ptr[t + 1];
    // this block's part of the tiles: the parts that hold the rows' own
    // columns, and with them the expensive pairs, are the first of the grid
    // to start
    int part = blockIdx.y;
    if (gridDim.y > 1) {
        int lo = run0, hi = run1 - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.N.runs[mid].x <= e0) lo = mid;
            else hi = mid - 1;
        }
        const int64_t own = (a.N.runs[lo].y + (e0 - a.N.runs[lo].x)) / cols;
        part = (int)((part + max((int64_t)0, min(own, (int64_t)ntile - 1)) * gridDim.y / ntile) % gridDim.y);
    }
    const int tb = (int)((int64_t)ntile * part / gridDim.y), te = (int)((int64_t)ntile * (part + 1) / gridDim.y);
    unsigned pend = 0;                                 // columns of this lane that found the queue full
    for (int tile = tb;; ++tile) {
        // the queue is worked off after the last tile, before one that may fill
        // it, and where it was too short for the last one (s_qn is the same in
        // every thread: no pushes since the barrier)
        for (;;) {
            const bool full = __syncthreads_or(pend != 0);
            if (!full && (tile < te ? s_qn <= kFusedQueue / 2 : s_qn == 0)) break;
            drain();
            __syncthreads();
            if (!full) break;
            for (unsigned left = pend; left; left &= left - 1) {
                const int b = __ffs((int)left) - 1, slot = atomicAdd(&s_qn, 1);
                if (slot >= kFusedQueue) break;
                s_qj[slot] = s_j[warp * chunk + b];
                s_qr[slot] = (unsigned char)rr;
                pend &= ~(1u << b);
            }
        }
        if (tile >= te) break;
        bool q_here = false;
        {
            const int p = tile * cols + threadIdx.x;
            if ((int)threadIdx.x < cols && p < nc) {
                int lo = run0, hi = run1 - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (a.N.runs[mid].y <= p) lo = mid;
                    else hi = mid - 1;
                }
                const int2 rn = a.N.runs[lo];
                const int j = rn.x + (p - rn.y);
                const float4 h = a.E.chi[j];
                float4 l = a.E.clo[j];
                l.w = __frcp_rn(h.w);
                s_hi[threadIdx.x] = h;
                s_lo[threadIdx.x] = l;
                s_n[threadIdx.x] = a.E.nrm[j];
                s_j[threadIdx.x] = j;
                if (!kT) {
                    s_va[threadIdx.x] = a.E.va[j];
                    s_e1[threadIdx.x] = a.E.e1[j];
                    s_e2[threadIdx.x] = a.E.e2[j];
                    float2 cp = a.cp[j], cq = a.cq[j];
                    if (kFold) {
                        const float2 xv = x[j];
                        cp = cmul(cp, xv);
                        cq = cmul(cq, xv);
                    }
                    s_c[threadIdx.x] = make_float4(cp.x, cp.y, cq.x, cq.y);
                    q_here = cq.x != 0.f || cq.y != 0.f;
                }
                if (!kFold)
#pragma unroll
                    for (int r = 0; r < NR; ++r) s_x[r][threadIdx.x] = x[r * a.E.n + j];
            }
        }
        const bool q_tile = __syncthreads_or(q_here);
        if (!kT) needq = q_tile;
        const int c0 = warp * chunk, c1 = min(c0 + chunk, nc - tile * cols);
        // the tile's own sum first: a long row's sum is then one of few terms
        float2 ta[NR], tq = make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < NR; ++r) ta[r] = make_float2(0.f, 0.f);
        for (int cb = c0; cb < c1; cb += R) {
            const int c = cb + sub;
            if (!live || c >= c1) continue;
            const float4 whi = s_hi[c], wlo = s_lo[c];
            float3 D0;                                  // x_j - x_i
            const float rt2 = kT ? pair_rt2(f3(ehi), f3(elo), f3(whi), f3(wlo), einv, D0)
                                 : pair_rt2(f3(whi), f3(wlo), f3(ehi), f3(elo), wlo.w, D0);
            int code = 0;
            if (rt2 > rt1) code = 1;
            else if (rt2 > rth && rt2 < rt1lo && (rt2 > rt2hi || rt2 < rt2lo)) code = rt2 > rt2hi ? 2 : 3;
            const float3 wn = f3(s_n[c]);
            const float3 nx = kT ? wn : f3(en), ny = kT ? f3(en) : wn;
            const float area = kT ? ehi.w : whi.w;
            if (code == 0) {
                if (s_j[c] == (int)e) {
                    s_self[rr] = 1;
                    continue;
                }
                const int slot = atomicAdd(&s_qn, 1);
                if (slot < kFusedQueue) {
                    s_qj[slot] = s_j[c];
                    s_qr[slot] = (unsigned char)rr;
                } else {
                    pend |= 1u << (c - c0);
                }
                continue;
            }
            float2 Kp = make_float2(0.f, 0.f), Kq = Kp;
            if (code == 1) {
                // the 1 x 1 conical rule is the centroid rule
                bm_point_sel(D0, nx, ny, k, ik_inv, area, needp, needq, Kp, Kq);
            } else {
                const float3 g1 = kT ? ee1 : f3(s_e1[c]), g2 = kT ? ee2 : f3(s_e2[c]);
                const float3 base = add3(D0, kT ? eva : f3(s_va[c]));
                const int u1 = code == 2 ? 5 : 14;
                for (int u = code == 2 ? 1 : 5; u < u1; ++u) {
                    const float4 rl = s_rule[u];
                    bm_point_sel(mad3(rl.y, g2, mad3(rl.x, g1, base)), nx, ny, k, ik_inv, area * rl.z, needp, needq, Kp,
                                 Kq);
                }
            }
            if (kT) {
                const float2 xv = s_x[0][c];
                ta[0] = cfma(Kp, xv, ta[0]);
                tq = cfma(Kq, xv, tq);
            } else {
                const float4 cc = s_c[c];
                if (kFold) {
                    ta[0] = cfma(Kp, make_float2(cc.x, cc.y), ta[0]);
                    if (needq) ta[0] = cfma(Kq, make_float2(cc.z, cc.w), ta[0]);
                } else {
                    float2 v = cmul(make_float2(cc.x, cc.y), Kp);
                    if (needq) v = cfma(make_float2(cc.z, cc.w), Kq, v);
#pragma unroll
                    for (int r = 0; r < NR; ++r) ta[r] = cfma(v, s_x[r][c], ta[r]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] = cadd(acc[r], ta[r]);
        accq = cadd(accq, tq);
    }
    if (kT) acc[0] = cadd(cmul(ecp, acc[0]), cmul(ecq, accq));
    for (int row = warp; row < cnt; row += kW) {       // the self terms
        if (!s_self[row]) continue;
        const int64_t j = e0 + row;
        float2 G, Ee;
        self_points(a.E, j, k, Q, lane, G, Ee);
        G = warp_sum(G);
        Ee = warp_sum(Ee);
        if (lane == 0) add_entry<NR>(&s_h[0][row], x, a.E.n, j, self_entry(G, Ee, k, ik_inv, a.tau, a.cp[j], a.cq[j]));
    }
    // the sums of a row: columns side by side in a warp, then the warps in order
    float2 *red = reinterpret_cast<float2 *>(s_buf);
    float2 *dst = out + (int64_t)part * NR * a.E.n;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        __syncthreads();
        red[threadIdx.x] = lanes_sum(acc[r], w);
        __syncthreads();
        if (threadIdx.x < cnt) {
            Sum2 v(s_h[r][threadIdx.x]);
            for (int q = 0; q < kW; ++q) v.add(red[q * 32 + threadIdx.x]);
            dst[r * a.E.n + e0 + threadIdx.x] = v.value();
        }
    }
}

#define BEM_FUSED_KERNEL(NAME, NR, T)                                                                                \
    __global__ void __launch_bounds__(kFusedThreads, 4)                                                             \
        NAME(NearArgs a, const int4 *__restrict__ tasks, int rows, int cols, const float2 *__restrict__ x,          \
             float2 *__restrict__ out, int *__restrict__ err, const int *skip)                                      \
    {                                                                                                                \
        if (skip_now(skip)) return;                                                                                  \
        near_fused_body<NR, T>(a, tasks, rows, cols, x, out, err);                                                               \
    }
BEM_FUSED_KERNEL(k_near_fused_1, 1, false)
BEM_FUSED_KERNEL(k_near_fused_2, 2, false)
BEM_FUSED_KERNEL(k_near_fused_4, 4, false)
BEM_FUSED_KERNEL(k_near_fused_t, 1, true)
#undef BEM_FUSED_KERNEL

// y = the S column parts of a recomputed product (part[s][n] with n the rows
// of every plane) in order.
__global__ void k_near_fused_sum(const float2 *__restrict__ part, int S, int64_t n, float2 *__restrict__ y,
                                 const int *skip)
{
    if (skip_now(skip)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    Sum2 v;
#pragma unroll 4
    for (int s = 0; s < S; ++s) v.add(part[(int64_t)s * n + i]);
    y[i] = v.value();
}

// Row scaling of Eq. SystemI (Sec. 3.2, the solver's row-scaling
// preconditioner): dinv_i = 1 / A_ii, the self entry of row i with the
// element's own column coefficients (the value the stored near field holds).
__global__ void k_row_scale_init(NearArgs a, float2 *__restrict__ dinv, int *__restrict__ err)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.E.n) return;
    const float4 ch = a.E.chi[i], cl = a.E.clo[i];
    const float3 xhi = f3(ch), xlo = f3(cl), nx = f3(a.E.nrm[i]);
    const double xd[3] = {a.E.cd[3 * i], a.E.cd[3 * i + 1], a.E.cd[3 * i + 2]};
    float2 v;
    if (!bm_entry(a.E, i, i, xhi, xlo, xd, nx, a.k, a.ik_inv, a.tau, *a.Q, a.cp[i], a.cq[i], v)) {
        atomicMin(err, (int)i);
        v = make_float2(1.f, 0.f);
    }
    const float m2 = v.x * v.x + v.y * v.y;
    dinv[i] = m2 > 0.f ? make_float2(v.x / m2, -v.y / m2) : make_float2(1.f, 0.f);
}

// y_i *= dinv_i, and y2_i *= dinv_i when y2 is given (the two parts of a
// product that the Gram-Schmidt step adds): the row scaling of a product or
// of the right-hand side.  Skips with the product kernels.
__global__ void k_row_scale(float2 *__restrict__ y, float2 *__restrict__ y2, const float2 *__restrict__ dinv,
                            int64_t n, const int *skip)
{
    if (skip_now(skip)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float2 d = dinv[i];
    const int64_t q = (int64_t)blockIdx.y * n + i;         // the right-hand side's plane
    y[q] = cmul(y[q], d);
    if (y2) y2[q] = cmul(y2[q], d);
}

// Block-Jacobi preconditioner (the block form of the solver's row scaling,
// Sec. 3.2): P = inverse of the block diagonal of A over sub-blocks of at
// most kBjMax consecutive elements of one leaf (blocks[b] = (first element,
// size, offset of its inverse, 0)).  One CUDA block per sub-block: the
// entries A_ij of the sub-block, read from the stored near field (val; a leaf
// is in its own near list) or, without one (val null), by bm_entry, the same
// values (a sub-block's pairs are the subdivided and self terms: computing
// them took 613 us on 13,520 elements, reading them 84);
// then Gauss-Jordan inversion in place with partial pivoting in shared
// memory (FP32 complex).  The inverse is stored column-major so that the
// apply kernel's threads (one per row) read consecutive entries.  A zero
// pivot leaves the sub-block's inverse the identity (no preconditioning
// there); err takes the subdivision limit of the entries, as for the stored
// near field.
__global__ void __launch_bounds__(256) k_bj_factor(NearArgs a, const int4 *__restrict__ blocks,
                                                   const float2 *__restrict__ val, float2 *__restrict__ binv,
                                                   int *__restrict__ err)
{
    __shared__ float2 A[kBjMax][kBjMax + 1];
    __shared__ int piv[kBjMax];
    __shared__ int s_p;
    __shared__ bool s_bad;
    const int4 B = blocks[blockIdx.x];
    const int64_t e0 = B.x;
    const int nb = B.y;
    const QuadTables &Q = *a.Q;
    // position of column e0 in the rows of this leaf (val)
    int64_t col0 = 0;
    if (val) {
        const int t = a.N.leaf_of[e0];
        int lo = a.N.run_ptr[t], hi = a.N.run_ptr[t + 1] - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.N.runs[mid].x <= e0) lo = mid;
            else hi = mid - 1;
        }
        col0 = a.N.runs[lo].y + (e0 - a.N.runs[lo].x);
    }
    for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
        const int r = idx / nb, c = idx % nb;
        const int64_t i = e0 + r, j = e0 + c;
        if (val) {
            A[r][c] = val[a.N.row_ptr[i] + col0 + c];
            continue;
        }
        const float4 ch = a.E.chi[i], cl = a.E.clo[i];
        const double xd[3] = {a.E.cd[3 * i], a.E.cd[3 * i + 1], a.E.cd[3 * i + 2]};
        float2 v;
        if (!bm_entry(a.E, i, j, f3(ch), f3(cl), xd, f3(a.E.nrm[i]), a.k, a.ik_inv, a.tau, Q, a.cp[j], a.cq[j], v)) {
            atomicMin(err, (int)j);
            v = make_float2(r == c ? 1.f : 0.f, 0.f);
        }
        A[r][c] = v;
    }
    if (threadIdx.x == 0) s_bad = false;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < nb; ++k) {
        // pivot: the largest |A[i][k]|, i >= k (warp 0)
        if (warp == 0) {
            float best = -1.f;
            int bi = k;
            for (int i = k + lane; i < nb; i += 32) {
                const float m = A[i][k].x * A[i][k].x + A[i][k].y * A[i][k].y;
                if (m > best) { best = m; bi = i; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (lane == 0) {
                s_p = bi;
                piv[k] = bi;
                if (!(best > 0.f)) s_bad = true;
            }
        }
        __syncthreads();
        if (s_bad) break;
        const int p = s_p;
        if (p != k)
            for (int c = threadIdx.x; c < nb; c += blockDim.x) {
                const float2 t = A[k][c];
                A[k][c] = A[p][c];
                A[p][c] = t;
            }
        __syncthreads();
        const float2 d = A[k][k];
        const float dm = 1.f / (d.x * d.x + d.y * d.y);
        const float2 inv = make_float2(d.x * dm, -d.y * dm);
        __syncthreads();
        // row k /= pivot (the pivot's own place becomes 1 / pivot)
        for (int c = threadIdx.x; c < nb; c += blockDim.x) A[k][c] = c == k ? inv : cmul(A[k][c], inv);
        __syncthreads();
        // eliminate column k from the other rows (their column k becomes -f / pivot)
        for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
            const int i = idx / nb, c = idx % nb;
            if (i == k) continue;
            const float2 f = A[i][k];
            if (c == k) continue;
            A[i][c] = csub(A[i][c], cmul(f, A[k][c]));
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nb; i += blockDim.x)
            if (i != k) A[i][k] = make_float2(-(A[i][k].x * inv.x - A[i][k].y * inv.y),
                                              -(A[i][k].x * inv.y + A[i][k].y * inv.x));
        __syncthreads();
    }
    if (s_bad) {
        for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x)
            binv[B.z + idx] = make_float2((idx / nb) == (idx % nb) ? 1.f : 0.f, 0.f);
        return;
    }
    // undo the row exchanges as column exchanges, last first
    for (int k = nb - 1; k >= 0; --k) {
        const int p = piv[k];
        if (p != k)
            for (int r = threadIdx.x; r < nb; r += blockDim.x) {
                const float2 t = A[r][k];
                A[r][k] = A[r][p];
                A[r][p] = t;
            }
        __syncthreads();
    }
    for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
        const int c = idx / nb, r = idx % nb;      // column-major
        binv[B.z + idx] = A[r][c];
    }
}

// w <- P (w + wnear) over the sub-blocks (wnear, when given, is cleared):
// the preconditioner applied to a product whose two parts the Gram-Schmidt
// step would add, or to a right-hand side / residual (wnear null).  One block
// of kBjMax threads per sub-block, one thread per row.  Skips with the
// product kernels.
__global__ void __launch_bounds__(kBjMax) k_bj_apply(const int4 *__restrict__ blocks, const float2 *__restrict__ binv,
                                                     float2 *__restrict__ w, float2 *__restrict__ wnear,
                                                     int64_t n, const int *skip)
{
    if (skip_now(skip)) return;
    __shared__ float2 xs[kBjMax];
    const int4 B = blocks[blockIdx.x];
    const int nb = B.y;
    const int r = threadIdx.x;
    const int64_t o = (int64_t)blockIdx.y * n + B.x + r;   // the row in its right-hand side's plane
    if (r < nb) {
        float2 v = w[o];
        if (wnear) v = cadd(v, wnear[o]);
        xs[r] = v;
    }
    __syncthreads();
    if (r >= nb) return;
    const float2 *__restrict__ col = binv + B.z + r;
    float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
    // eight columns' loads in flight per thread (the inverses come from L2 or
    // HBM and a leaf's block is a few such batches: the kernel is their latency)
    int c = 0;
    for (; c + 8 <= nb; c += 8, col += 8 * nb) {
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = col[u * nb];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            acc0 = cfma(v[u], xs[c + u], acc0);
            acc1 = cfma(v[u + 1], xs[c + u + 1], acc1);
        }
    }
    for (; c + 1 < nb; c += 2, col += 2 * nb) {
        acc0 = cfma(col[0], xs[c], acc0);
        acc1 = cfma(col[nb], xs[c + 1], acc1);
    }
    if (c < nb) acc0 = cfma(col[0], xs[c], acc0);
    w[o] = cadd(acc0, acc1);
    if (wnear) wnear[o] = make_float2(0.f, 0.f);
}

// ------------------------------------------------------------------ adjoint
// Inputs of the transposed product's far field.  With the antipodal
// symmetry of the sphere grid and D(-X, s) = D(X, -s) (Eq. FMMBase), the far
// part of A^T x is the forward aggregation of the weights (alpha, c) =
// (x_i, -x_i) (row operator 1 - s.n_i on the source side), the forward
// transfer, and a disaggregation with the row factor A_i (cq_i - ik cp_i
// (s.n_i)) = a_i + b_i (s.n_i) (the column factor of the forward product).
// x: internal order, or null to use x_int as it stands.
__global__ void k_prep_t(int64_t n, const float2 *__restrict__ x, float2 *__restrict__ xint,
                         float4 *__restrict__ wts, float4 *__restrict__ rowf, const float4 *__restrict__ chi,
                         const float2 *__restrict__ cp, const float2 *__restrict__ cq, float k, const int *skip)
{
    if (skip_now(skip)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float2 xv = x ? x[i] : xint[i];
    if (x) xint[i] = xv;
    if (wts) wts[i] = make_float4(xv.x, xv.y, -xv.x, -xv.y);
    const float A = chi[i].w;
    const float2 av = cscale(cq[i], A), t = cscale(cp[i], A);
    rowf[i] = make_float4(av.x, av.y, k * t.y, -k * t.x);   // (A cq, -ik A cp)
}

// Transposed field operator of the representation formula (Eq. BIE_I with
// lambda = 1, the element rules of k_field): for each element j,
//   g_j = sum_m G(x_m)_j conj(f_m),  h_j = sum_m H(x_m)_j conj(f_m),
// and the adjoint right-hand side r_j = cp_j h_j - cq_j g_j (the column
// coefficients carry tau, so r = F^T conj(f) with F the map from the
// unknowns to the field).  One warp per element, lanes over the points.
__global__ void k_field_t(ElemDev E, const QuadTables *__restrict__ Qp, const double *__restrict__ pts, int64_t M,
                          float k, const float2 *__restrict__ f, const float2 *__restrict__ cp,
                          const float2 *__restrict__ cq, float2 *__restrict__ g_out, float2 *__restrict__ r_out,
                          int *err)
{
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (j >= E.n) return;
    const QuadTables &Q = *Qp;
    float2 ga = make_float2(0.f, 0.f), ha = make_float2(0.f, 0.f);
    for (int64_t m = lane; m < M; m += 32) {
        const double xd[3] = {pts[3 * m], pts[3 * m + 1], pts[3 * m + 2]};
        const float3 xhi = make_float3((float)xd[0], (float)xd[1], (float)xd[2]);
        const float3 xlo = make_float3((float)(xd[0] - (double)xhi.x), (float)(xd[1] - (double)xhi.y),
                                       (float)(xd[2] - (double)xhi.z));
        float2 G = make_float2(0.f, 0.f), H = make_float2(0.f, 0.f);
        if (!integrate_regular<true>(E, j, xhi, xlo, xd, make_float3(0.f, 0.f, 1.f), k, 1.0f / k, Q, G, H)) {
            atomicMin(err, (int)j);
            continue;
        }
        const float2 w = make_float2(f[m].x, -f[m].y);
        ga = cfma(G, w, ga);
        ha = cfma(H, w, ha);
    }
    ga = warp_sum(ga);
    ha = warp_sum(ha);
    if (lane == 0) {
        g_out[j] = ga;
        r_out[j] = csub(cmul(cp[j], ha), cmul(cq[j], ga));
    }
}

// Gradient of L = sum_m |f_m|^2 with respect to the region admittances Y_r,
// from the forward solution u, the adjoint solution lambda of
// A^T lambda = F^T conj(f), g = G_f^T conj(f) and aq = A_q^T lambda (A_q the
// operator on q-unknowns, c^p = 0 and c^q = 1): element j of region r adds
//   t_j = d u_j (-tau g_j - aq_j),  d = dc^q_j / dY_r = -tau i k rho c,
// and grad_r = 2 conj(sum_j t_j) = dL/dRe Y_r + i dL/dIm Y_r.  acc
// (zeroed by the caller): [n_regions][2] gradient, then L.  region: per
// element (internal order), -1 when the element is not ADMI.
__global__ void k_adjoint_reduce(const float2 *__restrict__ u, const float2 *__restrict__ g,
                                 const float2 *__restrict__ aq, const int *__restrict__ region, int64_t n,
                                 float tau, double dre, double dim, const float2 *__restrict__ f, int64_t M,
                                 int nreg, double *acc)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const int r = region[i];
        if (r >= 0 && r < nreg) {
            const double gr = g[i].x, gi = g[i].y, ar = aq[i].x, ai = aq[i].y;
            const double br = -tau * gr - ar, bi = -tau * gi - ai;      // -tau g_j - aq_j
            const double ur = u[i].x, ui = u[i].y;
            const double cr = ur * br - ui * bi, ci = ur * bi + ui * br; // u_j (...)
            const double tr = dre * cr - dim * ci, ti = dre * ci + dim * cr;
            atomicAdd(&acc[2 * r], 2.0 * tr);
            atomicAdd(&acc[2 * r + 1], -2.0 * ti);
        }
    }
    if (i < M) {
        const double fr_ = f[i].x, fi = f[i].y;
        atomicAdd(&acc[2 * nreg], fr_ * fr_ + fi * fi);
    }
}

// ------------------------------------------------------------------ far field
// Per product: gather x into the internal order (x_int[i] = x[perm[i]] or
// x = xbase + jidx * n) and form the aggregation weights of the centroid
// rule, alpha_i = A_i cq_i x_i and c_i = ik A_i cp_i x_i, so that the column
// factor of Sec. 3.3.1 is alpha_i + c_i (n_i . s).
__device__ __forceinline__ void prep_store(const PrepArgs &a, int64_t i, float2 xv)
{
    a.xint[i] = xv;
    if (a.wts) {
        const float A = a.chi[i].w;
        const float2 al = cscale(cmul(a.cq[i], xv), A);
        const float2 t = cscale(cmul(a.cp[i], xv), A);
        // (alpha, c) = (A cq x, ik A cp x)
        a.wts[i] = make_float4(al.x, al.y, -a.k * t.y, a.k * t.x);
    }
}
__global__ void k_prep(PrepArgs a, const int *skip)
{
    if (skip_now(skip)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    const float2 *xb = a.x;
    if (a.jidx) xb += (int64_t)(*a.jidx) * a.n;
    if (blockIdx.y) {
        // right-hand side blockIdx.y: its planes of x, xint and wts
        const int64_t o = (int64_t)blockIdx.y * a.plane;
        xb += (int64_t)blockIdx.y * a.xplane;
        a.xint += o;
        if (a.wts) a.wts += o;
    }
    prep_store(a, i, a.perm ? xb[a.perm[i]] : xb[i]);
}

// Streamed 8-byte load of a stored phase (read once per product): read-only
// path, no L1 allocation.
__device__ __forceinline__ float2 ld_stream2(const float2 *p)
{
    float2 v;
    asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

// Aggregation (Sec. 3.3.3, matrix T(l) with the centroid rule): for every
// source cluster c and direction s_nu,
//   M_c(nu) = sum_{j in c} e^{ik (z_c - x_j).s_nu} (alpha_j + c_j (n_j . s_nu)).
// One block per task: a chunk of at most kAggChunk elements of one cluster
// and kAggThreads antipodal direction pairs, one pair per thread; phases in
// turns, regenerated (kTab false) or read from the level's stored phases
// (kTab, the same values: k_phase_table evaluates the same expression).
// Bound by FP32 issue: about 14 instructions of phase and s.n per pair, and the
// sums.  These are kept as four real-weighted sums per right-hand side,
// S1 = sum cs alpha, S2 = sum sn alpha, S3 = sum cs t c, S4 = sum sn t c (two
// operations each per pair), from which both directions follow at the end:
//   M(s) = S1 + S3 + i (S2 + S4),  M(-s) = S1 - S3 - i (S2 - S4);
// forming alpha +- t c per pair took twelve.  A chunk whose alpha (no q on any
// of its elements: a sound-hard surface) or c (pressure given) are all zero
// leaves out their two sums.  Four right-hand sides on 158,420 elements: 602 ->
// 391 us; one on 20,480: 18.3 -> 16.4 us.
// Tasks of equal size keep every block short, so no large cluster sets the
// kernel's length.  For a cluster split into several element chunks, the
// last of its blocks to finish sums the chunks' partial rows in row order.
template <int NR, bool kTab>
__device__ __forceinline__ void aggregate_body(const LevelsArgs &A, const float4 *__restrict__ wts,
                                               int64_t wplane, const float4 *__restrict__ nrm)
{
    const AggTask T = A.tasks[blockIdx.x];
    const FarArgs &f = A.lev[T.lev];
    __shared__ float4 sd[kTab ? 1 : kAggChunk];   // (z_c - x_j) k / (2 pi)
    __shared__ float4 sw[NR][kAggChunk];           // (alpha_j, c_j) per right-hand side
    __shared__ float4 sn[kAggChunk];               // n_j
    const float kt = f.k * 0.15915494309189535f;
    int parts = 0;                                 // bit 0: some alpha, bit 1: some c
    for (int q = threadIdx.x; q < T.ne; q += blockDim.x) {
        const int64_t j = T.e0 + q;
        if (!kTab) {
            const float4 d = f.dz[j];
            sd[q] = make_float4(kt * d.x, kt * d.y, kt * d.z, 0.f);
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const float4 w = wts[r * wplane + j];
            sw[r][q] = w;
            parts |= (w.x != 0.f || w.y != 0.f ? 1 : 0) | (w.z != 0.f || w.w != 0.f ? 2 : 0);
        }
        sn[q] = nrm[j];
    }
    const bool has_a = __syncthreads_or(parts & 1), has_c = __syncthreads_or(parts & 2);
    // directions in antipodal halves: s_{p + h} = -s_p, so one phase serves
    // both, e^{ik d.(-s)} = conj(e^{ik d.s}), and n.(-s) = -(n.s)
    float2 *__restrict__ out = f.M + (int64_t)T.row * f.nd;
    const int h = f.nd / 2;
    const int p = T.p0 + threadIdx.x;
    if (p < h) {
        const float4 sv = f.dirs[p];
        float2 s1[NR], s2[NR], s3[NR], s4[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) s1[r] = s2[r] = s3[r] = s4[r] = make_float2(0.f, 0.f);
        auto run = [&](auto with_a, auto with_c) {
            constexpr bool kA = decltype(with_a)::value, kC = decltype(with_c)::value;
            // element q of the chunk with the phase cs0 + i sn0
            auto term = [&](int q, float sn0, float cs0) {
                float ct = 0.f, st = 0.f;
                if (kC) {
                    const float4 n = sn[q];
                    const float t = fmaf(n.x, sv.x, fmaf(n.y, sv.y, n.z * sv.z));
                    ct = cs0 * t;
                    st = sn0 * t;
                }
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const float4 w = sw[r][q];
                    if (kA) {
                        s1[r] = make_float2(fmaf(cs0, w.x, s1[r].x), fmaf(cs0, w.y, s1[r].y));
                        s2[r] = make_float2(fmaf(sn0, w.x, s2[r].x), fmaf(sn0, w.y, s2[r].y));
                    }
                    if (kC) {
                        s3[r] = make_float2(fmaf(ct, w.z, s3[r].x), fmaf(ct, w.w, s3[r].y));
                        s4[r] = make_float2(fmaf(st, w.z, s4[r].x), fmaf(st, w.w, s4[r].y));
                    }
                }
            };
            if (kTab) {
                // the chunk's rows of stored phases, 16 loads per thread in flight
                const float2 *__restrict__ ph = f.ph + (int64_t)T.e0 * f.phs + p;
                int q = 0;
                for (; q + 16 <= T.ne; q += 16) {
                    float2 e[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) e[u] = ld_stream2(ph + (int64_t)(q + u) * f.phs);
#pragma unroll
                    for (int u = 0; u < 16; ++u) term(q + u, e[u].y, e[u].x);
                }
                for (; q < T.ne; ++q) {
                    const float2 e = ld_stream2(ph + (int64_t)q * f.phs);
                    term(q, e.y, e.x);
                }
            } else {
                for (int q = 0; q < T.ne; ++q) {
                    const float4 d = sd[q];
                    float sn0, cs0;
                    sincos_turns(fmaf(d.x, sv.x, fmaf(d.y, sv.y, d.z * sv.z)), &sn0, &cs0);
                    term(q, sn0, cs0);
                }
            }
        };
        if (has_a && has_c) run(std::true_type(), std::true_type());
        else if (has_c) run(std::false_type(), std::true_type());
        else if (has_a) run(std::true_type(), std::false_type());
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            out[r * f.mplane + p] = make_float2((s1[r].x + s3[r].x) - (s2[r].y + s4[r].y),
                                                (s1[r].y + s3[r].y) + (s2[r].x + s4[r].x));
            out[r * f.mplane + p + h] = make_float2((s1[r].x - s3[r].x) + (s2[r].y - s4[r].y),
                                                    (s1[r].y - s3[r].y) - (s2[r].x - s4[r].x));
        }
    }
    aggregate_reduce(A, T, f, kAggThreads, NR);
}

#define BEM_AGGREGATE_KERNEL(NR, TAB, NAME)                                                                           \
    __global__ void __launch_bounds__(kAggThreads)                                                                   \
        NAME(const __grid_constant__ LevelsArgs A, const float4 *__restrict__ wts, int64_t wplane,                    \
             const float4 *__restrict__ nrm, const int *skip)                                                        \
    {                                                                                                                 \
        if (skip_now(skip)) return;                                                                                   \
        aggregate_body<NR, TAB>(A, wts, wplane, nrm);                                                                \
    }
BEM_AGGREGATE_KERNEL(1, false, k_aggregate_1)
BEM_AGGREGATE_KERNEL(2, false, k_aggregate_2)
BEM_AGGREGATE_KERNEL(3, false, k_aggregate_3)
BEM_AGGREGATE_KERNEL(4, false, k_aggregate_4)
BEM_AGGREGATE_KERNEL(1, true, k_aggregate_1t)
#undef BEM_AGGREGATE_KERNEL

// Stored phases of the aggregation (and, conjugated, of the
// disaggregation) for every level, element and antipodal direction pair,
// by the expression the products evaluate when they regenerate them:
// ph[j][p] = (cos, sin) 2 pi t, t = (k / 2 pi)(z_c - x_j).s_p in turns;
// the padding column of odd rows holds zero.
__global__ void k_phase_table(PhaseTableArgs a)
{
    int l = 0;
    while (l + 1 < a.nlev && (int)blockIdx.x >= a.start[l + 1]) ++l;
    const PhaseLevel &L = a.lev[l];
    const int64_t e0 = (int64_t)((int)blockIdx.x - a.start[l]) * kPhaseElems;
    const float kt = a.k * 0.15915494309189535f;
    for (int p = threadIdx.x; p < L.phs; p += blockDim.x) {
        const float4 sv = p < L.h ? L.dirs[p] : make_float4(0.f, 0.f, 0.f, 0.f);
        for (int u = 0; u < kPhaseElems; ++u) {
            const int64_t j = e0 + u;
            if (j >= a.n) break;
            float2 v = make_float2(0.f, 0.f);
            if (p < L.h) {
                const float4 d = L.dz[j];
                const float dx = kt * d.x, dy = kt * d.y, dzz = kt * d.z;
                float sn0, cs0;
                sincos_turns(fmaf(dx, sv.x, fmaf(dy, sv.y, dzz * sv.z)), &sn0, &cs0);
                v = make_float2(cs0, sn0);
            }
            L.ph[j * L.phs + p] = v;
        }
    }
}

// sin / cos of 2 pi x by sincos_turns and by sincospif, for the unit tests.
__global__ void k_selftest_sincos(const float *__restrict__ x, int64_t n, float4 *__restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float s0, c0, s1, c1;
    sincos_turns(x[i], &s0, &c0);
    sincospif(2.f * x[i], &s1, &c1);
    out[i] = make_float4(s0, c0, s1, c1);
}

// Diagonal transfer (Sec. 3.3.3, matrix D(l)): for every target cluster t
// with an interaction list (Sec. 3.3.4),
//   Lambda_t(nu) = sum_{s in I(t)} D_L(z_t - z_s, s_nu) M_s(nu).
// A block takes one target and kTransferDirs directions, two per lane (one
// 16-byte load each of D and M per list entry); its kTransferWarps warps take
// every kTransferWarps-th list entry, each with kTransferUnroll entries in
// flight, and the partial sums are added in warp order.  Few warps per target
// with deep load batches hold fewer registers and warps of an SM for the same
// L2 traffic, which leaves room for the near-field product running beside.
// One direction per lane and two warps per target took 26.1 us on 20,480
// elements and 32.9 on 13,520; this 22.9 and 28.8 (two warps 22.0 and 30.9).
__global__ void __launch_bounds__(32 * kTransferWarps) k_transfer_split(const __grid_constant__ LevelsArgs A,
                                                                        const int *skip)
{
    if (skip_now(skip)) return;
    __shared__ float4 part[kTransferWarps][32];
    __shared__ int2 s_ent[kTransferEntries];      // (source cluster, offset) of the list entries
    const int4 T = A.tgroups[blockIdx.x];
    const FarArgs &f = A.lev[T.x];
    const int t = T.y, nu0 = T.z, nd = f.nd;
    // right-hand side blockIdx.y: its M and Lambda planes
    const float2 *__restrict__ Mp = f.M + blockIdx.y * f.mplane;
    float2 *__restrict__ Lp = f.Lam + blockIdx.y * f.lplane;
    const float2 *__restrict__ D = f.D;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nu = nu0 + 2 * lane;                // nd is even: a pair of directions is in range or not
    const bool live = nu < nd;
    const int b = f.il_ptr[t], e = f.il_ptr[t + 1];
    float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
    constexpr int kW = kTransferWarps, kU = kTransferUnroll;
    for (int c0 = b; c0 < e; c0 += kTransferEntries) {
        const int cnt = min(kTransferEntries, e - c0);
        __syncthreads();
        for (int q = threadIdx.x; q < cnt; q += blockDim.x)
            s_ent[q] = make_int2(f.il_src[c0 + q], f.il_off[c0 + q]);
        __syncthreads();
        if (!live) continue;
        int q = warp;
        for (; q + kW * (kU - 1) < cnt; q += kW * kU) {
            float4 dv[kU], mv[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int2 en = s_ent[q + kW * u];
                dv[u] = __ldg(reinterpret_cast<const float4 *>(D + (int64_t)en.y * nd + nu));
                mv[u] = *reinterpret_cast<const float4 *>(Mp + (int64_t)en.x * nd + nu);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                acc0 = cfma(make_float2(dv[u].x, dv[u].y), make_float2(mv[u].x, mv[u].y), acc0);
                acc1 = cfma(make_float2(dv[u].z, dv[u].w), make_float2(mv[u].z, mv[u].w), acc1);
            }
        }
        for (; q < cnt; q += kW) {
            const int2 en = s_ent[q];
            const float4 dv = __ldg(reinterpret_cast<const float4 *>(D + (int64_t)en.y * nd + nu));
            const float4 mv = *reinterpret_cast<const float4 *>(Mp + (int64_t)en.x * nd + nu);
            acc0 = cfma(make_float2(dv.x, dv.y), make_float2(mv.x, mv.y), acc0);
            acc1 = cfma(make_float2(dv.z, dv.w), make_float2(mv.z, mv.w), acc1);
        }
    }
    part[warp][lane] = make_float4(acc0.x, acc0.y, acc1.x, acc1.y);
    __syncthreads();
    if (warp == 0 && live) {
        float4 sum = part[0][lane];
#pragma unroll
        for (int w = 1; w < kW; ++w) {
            const float4 v = part[w][lane];
            sum = make_float4(sum.x + v.x, sum.y + v.y, sum.z + v.z, sum.w + v.w);
        }
        *reinterpret_cast<float4 *>(Lp + (int64_t)t * nd + nu) = sum;
    }
}

// The transfer for NR = 2 right-hand sides at once: the same blocks and list
// order as k_transfer_split, each D value loaded once for both planes (the
// M and Lambda planes are mplane and lplane apart).
template <int NR, int kW>
__device__ __forceinline__ void transfer_multi_body(const LevelsArgs &A)
{
    constexpr int kU = 8 / NR;
    __shared__ float2 part[NR][kW][32];
    __shared__ int2 s_ent[kTransferEntries];
    // a block takes half of a group of kTransferDirs directions (one per lane)
    const int4 T = A.tgroups[blockIdx.x >> 1];
    const FarArgs &f = A.lev[T.x];
    const int t = T.y, nu0 = T.z + 32 * (blockIdx.x & 1), nd = f.nd;
    const float2 *__restrict__ M = f.M, *__restrict__ D = f.D;
    const int64_t mplane = f.mplane;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nu = nu0 + lane;
    const bool live = nu < nd;
    if (nu0 >= nd) return;
    const int b = f.il_ptr[t], e = f.il_ptr[t + 1];
    float2 acc[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] = make_float2(0.f, 0.f);
    for (int c0 = b; c0 < e; c0 += kTransferEntries) {
        const int cnt = min(kTransferEntries, e - c0);
        __syncthreads();
        for (int q = threadIdx.x; q < cnt; q += blockDim.x)
            s_ent[q] = make_int2(f.il_src[c0 + q], f.il_off[c0 + q]);
        __syncthreads();
        if (!live) continue;
        int q = warp;
        for (; q + kW * (kU - 1) < cnt; q += kW * kU) {
            float2 dv[kU], mv[kU][NR];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int2 en = s_ent[q + kW * u];
                dv[u] = __ldg(D + (int64_t)en.y * nd + nu);
#pragma unroll
                for (int r = 0; r < NR; ++r) mv[u][r] = M[r * mplane + (int64_t)en.x * nd + nu];
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
#pragma unroll
                for (int r = 0; r < NR; ++r) acc[r] = cfma(dv[u], mv[u][r], acc[r]);
        }
        for (; q < cnt; q += kW) {
            const int2 en = s_ent[q];
            const float2 dv = __ldg(D + (int64_t)en.y * nd + nu);
#pragma unroll
            for (int r = 0; r < NR; ++r) acc[r] = cfma(dv, M[r * mplane + (int64_t)en.x * nd + nu], acc[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) part[r][warp][lane] = acc[r];
    __syncthreads();
    if (warp == 0 && live) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            float2 sum = part[r][0][lane];
#pragma unroll
            for (int w = 1; w < kW; ++w) sum = cadd(sum, part[r][w][lane]);
            f.Lam[r * f.lplane + (int64_t)t * nd + nu] = sum;
        }
    }
}

#define BEM_TRANSFER_MULTI_KERNEL(NAME, NR, W)                                                                        \
    __global__ void __launch_bounds__(32 * W) NAME(const __grid_constant__ LevelsArgs A, const int *skip)            \
    {                                                                                                                 \
        if (skip_now(skip)) return;                                                                                   \
        transfer_multi_body<NR, W>(A);                                                                                \
    }
BEM_TRANSFER_MULTI_KERNEL(k_transfer_m2, 2, kTransferWarps)
BEM_TRANSFER_MULTI_KERNEL(k_transfer_m2s, 2, 1)
#undef BEM_TRANSFER_MULTI_KERNEL

// The merged lists of pairs of targets (FarArgs::pair), one block per pair: the
// sources that both list, then the first target's others, then the second's,
// each in list order.  Runs once per set of lists, 10^6 entries in tens of microseconds;
// built on the host, 158,420 elements took 9 ms.
__global__ void __launch_bounds__(128) k_pair_lists(const int *__restrict__ il_ptr, const int *__restrict__ il_src,
                                                    const int *__restrict__ il_off, int4 *__restrict__ pair,
                                                    int4 *__restrict__ ent)
{
    __shared__ int s_n[4];
    const int4 T = pair[2 * blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int a0 = il_ptr[T.x], a1 = il_ptr[T.x + 1];
    const int b0 = T.y >= 0 ? il_ptr[T.y] : 0, b1 = T.y >= 0 ? il_ptr[T.y + 1] : 0;
    // entries [c0, c1) of one list whose source is (both) or is not in [o0, o1)
    // of the other, appended at end
    int end = a0;
    auto append = [&](int c0, int c1, int o0, int o1, bool both, bool second) {
        for (int c = c0; c < c1; c += 128) {
            const int r = c + threadIdx.x, src = r < c1 ? il_src[r] : -1;
            int off = -1;
            for (int q = o0; q < o1; ++q)
                if (il_src[q] == src) off = il_off[q];
            const bool take = r < c1 && (off >= 0) == both;
            const unsigned m = __ballot_sync(0xffffffffu, take);
            if (lane == 0) s_n[warp] = __popc(m);
            __syncthreads();
            int pos = end + __popc(m & ((1u << lane) - 1u));
            for (int w = 0; w < 4; ++w) {
                if (w < warp) pos += s_n[w];
                end += s_n[w];
            }
            if (take) ent[pos] = second ? make_int4(src, -1, il_off[r], 0) : make_int4(src, il_off[r], off, 0);
            __syncthreads();
        }
    };
    append(a0, a1, b0, b1, true, false);
    const int both = end - a0;
    append(a0, a1, b0, b1, false, false);
    append(b0, b1, a0, a1, false, true);
    if (threadIdx.x == 0) {
        pair[2 * blockIdx.x] = make_int4(T.x, T.y, a0, both);
        pair[2 * blockIdx.x + 1] = make_int4(end - a0, 0, 0, 0);
    }
}

// The transfer for four right-hand sides at once.  Each D value serves all of
// them (the M and Lambda planes are mplane and lplane apart), so the bytes are
// mostly M's, 32 per list entry and direction.  A block therefore takes two
// targets, neighbours in Morton order that share most of their sources, and 32
// directions (lanes): a source's M is read once for both.  The sources of both
// come first, in a loop without tests, since issue (67% of the slots) is what
// bounds the kernel then.  kU sources in flight per warp at 72 registers, 28 warps
// per SM (three in flight spill, and take 1065 us at 80 registers or 841 at 96).  One target per block
// took 49.4 us on 10,580 elements and 942 on 158,420; pairs with every source
// tested 43.3 and 827; this 42.5 and 796.  (Groups of four targets need
// registers that cost more warps than the bytes they save; for two right-hand
// sides M weighs less, and pairs took 638 us against 575.)
template <int NR, int kW, int kU>
__device__ __forceinline__ void transfer_pairs_body(const LevelsArgs &A)
{
    __shared__ float2 part[kW][2][NR][32];
    __shared__ int4 s_ent[kTransferEntries];
    const int4 T = A.tpairs[blockIdx.x];
    const FarArgs &f = A.lev[T.x];
    const int nd = f.nd, nu = T.z + (threadIdx.x & 31);
    const float2 *__restrict__ M = f.M + nu, *__restrict__ D = f.D + nu;
    const int64_t mplane = f.mplane;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool live = nu < nd;
    const int b = f.pair[2 * T.y].z, eb = b + f.pair[2 * T.y].w, e = b + f.pair[2 * T.y + 1].x;
    float2 acc[2][NR];
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[g][r] = make_float2(0.f, 0.f);
    for (int c0 = b; c0 < e; c0 += kTransferEntries) {
        const int cnt = min(kTransferEntries, e - c0);
        __syncthreads();
        for (int q = threadIdx.x; q < cnt; q += 32 * kW) s_ent[q] = f.pair_ent[c0 + q];
        __syncthreads();
        if (!live) continue;
        int q = warp;
        const int nboth = min(cnt, eb - c0) - kW * (kU - 1);
#pragma unroll 1
        for (; q < nboth; q += kW * kU) {                // sources of both
            float2 mv[kU][NR], dv[kU][2];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int4 en = s_ent[q + kW * u];
#pragma unroll
                for (int r = 0; r < NR; ++r) mv[u][r] = M[r * mplane + (int64_t)en.x * nd];
                dv[u][0] = __ldg(D + (int64_t)en.y * nd);
                dv[u][1] = __ldg(D + (int64_t)en.z * nd);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
#pragma unroll
                for (int g = 0; g < 2; ++g)
#pragma unroll
                    for (int r = 0; r < NR; ++r) acc[g][r] = cfma(dv[u][g], mv[u][r], acc[g][r]);
        }
#pragma unroll 1
        for (; q < cnt; q += kW * kU) {
            float2 mv[kU][NR], dv[kU][2];
            int off[kU][2];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                off[u][0] = off[u][1] = -1;
                if (q + kW * u < cnt) {
                    const int4 en = s_ent[q + kW * u];
                    off[u][0] = en.y;
                    off[u][1] = en.z;
#pragma unroll
                    for (int r = 0; r < NR; ++r) mv[u][r] = M[r * mplane + (int64_t)en.x * nd];
#pragma unroll
                    for (int g = 0; g < 2; ++g)
                        if (off[u][g] >= 0) dv[u][g] = __ldg(D + (int64_t)off[u][g] * nd);
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
#pragma unroll
                for (int g = 0; g < 2; ++g)
                    if (off[u][g] >= 0)
#pragma unroll
                        for (int r = 0; r < NR; ++r) acc[g][r] = cfma(dv[u][g], mv[u][r], acc[g][r]);
        }
    }
    const int4 tg = f.pair[2 * T.y];                   // the second target may be absent (-1)
    {
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int r = 0; r < NR; ++r) part[warp][g][r][lane] = acc[g][r];
        __syncthreads();
        if (warp > 0) return;
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int r = 0; r < NR; ++r)
#pragma unroll
                for (int w = 1; w < kW; ++w) acc[g][r] = cadd(acc[g][r], part[w][g][r][lane]);
    }
    if (!live) return;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int t = g ? tg.y : tg.x;
        if (t < 0) continue;
#pragma unroll
        for (int r = 0; r < NR; ++r) f.Lam[r * f.lplane + (int64_t)t * nd + nu] = acc[g][r];
    }
}

#define BEM_TRANSFER_PAIRS_KERNEL(NAME, W)                                                                            \
    __global__ void __launch_bounds__(32 * W, 28 / W) NAME(const __grid_constant__ LevelsArgs A, const int *skip)            \
    {                                                                                                                 \
        if (skip_now(skip)) return;                                                                                   \
        transfer_pairs_body<4, W, 2>(A);                                                                              \
    }
BEM_TRANSFER_PAIRS_KERNEL(k_transfer_p4, kTransferWarps)
BEM_TRANSFER_PAIRS_KERNEL(k_transfer_p4s, kPairManyWarps)
#undef BEM_TRANSFER_PAIRS_KERNEL

// Disaggregation over all levels (Sec. 3.3.3, matrix S(l), with the
// Burton-Miller row operator 1 + s.n_i) and the sum with the near field
// (when ynear is given; else y receives the far part alone):
//   y_i = near_i + (ik/16 pi^2) sum_l sum_nu w_nu (1 + s_nu.n_i)
//                   e^{ik (x_i - z_t).s_nu} Lambda_t(nu),
// for NR right-hand sides at once (one phase per element and direction serves
// all of them; planes n apart in ynear and y, lplane apart in Lambda).
// One block of kDisThreads per task (at most kDisTask elements of one leaf;
// large leaves are split so that no block is much longer than the others).
// Element-major: thread t takes element t % cnt of the task and every nsl-th
// antipodal direction pair (s_p, -s_p) (one phase and its conjugate; nsl =
// kDisThreads / cnt slices).  The leaf shares its cluster at every level, so
// the direction pairs and the weighted rows (A, B) of every plane are staged
// in shared memory in chunks of kDisPairChunk pairs, level by level, and read
// by all the task's elements at once; each thread keeps its element's sums in
// registers, and the slices' sums are added in slice order.
// kRowF (NR = 1): the row factor a_i + b_i (s.n_i) with per-element (a, b) =
// a.rowf[i] in place of 1 + s.n_i (the transposed product: two sums per
// element, S0 = sum (1-part) and S1 = sum (s.n-part), combined as a S0 + b S1).
constexpr int kDisPairChunk = 256;
template <int NR, bool kRowF, bool kTab>
__device__ __forceinline__ void disaggregate_body(const DisaggArgs &a, const float2 *__restrict__ ynear,
                                                  float2 *__restrict__ y)
{
    static_assert(!kRowF || NR == 1, "the transposed product has one right-hand side");
    constexpr int kS = kRowF ? 2 : 1;           // sums per element and plane
    // pairs per staged chunk; with stored phases the chunk's rows of them
    // are staged too (row stride kChunk + 1: the 16 elements of a half-warp
    // read one pair's phases from distinct banks)
    constexpr int kChunk = kTab ? kDisTabChunk : kDisPairChunk;
    static_assert(!kTab || kDisTabChunk <= kDisThreads, "the phase staging takes one pair per thread");
    __shared__ float4 dir_s[kChunk];
    __shared__ float4 ab_s[NR][kChunk];
    __shared__ float2 ph_s[kTab ? kDisTask : 1][kTab ? kChunk + 1 : 1];
    __shared__ float2 red[kDisThreads][NR * kS];
    const int2 tk = a.tasks[blockIdx.x];
    const int64_t e0 = tk.x, e1 = tk.y;
    const int cnt = (int)min((int64_t)kDisTask, e1 - e0);   // the host makes tasks of 1..kDisTask elements
    if (cnt <= 0) return;
    const int nsl = kDisThreads / cnt;
    const int q = threadIdx.x % cnt, sl = threadIdx.x / cnt;
    const bool act = sl < nsl;
    const float4 n = a.nrm[e0 + q];
    float2 acc[NR * kS];
#pragma unroll
    for (int r = 0; r < NR * kS; ++r) acc[r] = make_float2(0.f, 0.f);
    for (int l = 0; l < a.nlev; ++l) {
        const FarArgs &f = a.lev[l];
        const int c = f.elem_cl[e0];
        if (f.il_ptr[c] == f.il_ptr[c + 1]) continue;   // no interaction list at this level
        const int h = f.nd / 2;
        const float kt = -f.k * 0.15915494309189535f;
        const float4 dz = kTab ? make_float4(0.f, 0.f, 0.f, 0.f) : f.dz[e0 + q];   // z_c - x_i
        const float dx = kt * dz.x, dy = kt * dz.y, dzz = kt * dz.z;
        for (int p0 = 0; p0 < h; p0 += kChunk) {
            const int np = min(kChunk, h - p0);
            __syncthreads();
            // per antipodal pair: s_p and, with lp = w Lambda(s_p), lm =
            // w Lambda(-s_p), A = lp + lm and B = lp - lm, so that
            // (1 + t) lp + (1 - t) lm = A + t B and (1 + t) lp - (1 - t) lm = B + t A
            for (int i = threadIdx.x; i < np; i += blockDim.x) {
                const float4 d = f.dirs[p0 + i];
                dir_s[i] = d;
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const float2 *__restrict__ src = f.Lam + r * f.lplane + (int64_t)c * f.nd;
                    const float2 lp = cscale(src[p0 + i], d.w), lm = cscale(src[p0 + i + h], d.w);
                    ab_s[r][i] = make_float4(lp.x + lm.x, lp.y + lm.y, lp.x - lm.x, lp.y - lm.y);
                }
            }
            if (kTab) {
                // the task's rows of the chunk's phases (coalesced along the pairs)
                const float2 *__restrict__ src = f.ph + e0 * f.phs + p0;
                // (np <= blockDim.x: one pair per thread, every row's load in flight together)
                if (threadIdx.x < np) {
                    float2 v[kDisTask];
#pragma unroll
                    for (int qq = 0; qq < kDisTask; ++qq)
                        if (qq < cnt) v[qq] = ld_stream2(src + (int64_t)qq * f.phs + threadIdx.x);
#pragma unroll
                    for (int qq = 0; qq < kDisTask; ++qq)
                        if (qq < cnt) ph_s[qq][threadIdx.x] = v[qq];
                }
            }
            __syncthreads();
            if (!act) continue;
            for (int i = sl; i < np; i += nsl) {
                const float4 sv = dir_s[i];
                float sn0, cs0;
                if (kTab) {
                    // the phase of (x_i - z_c).s is the conjugate of the stored one
                    const float2 e = ph_s[q][i];
                    cs0 = e.x;
                    sn0 = -e.y;
                } else {
                    sincos_turns(fmaf(dx, sv.x, fmaf(dy, sv.y, dzz * sv.z)), &sn0, &cs0);
                }
                const float tn = fmaf(n.x, sv.x, fmaf(n.y, sv.y, n.z * sv.z));
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const float4 ab = ab_s[r][i];
                    if (kRowF) {
                        // S0 += cs A + i sn B, S1 += t (cs B + i sn A)
                        acc[0].x = fmaf(cs0, ab.x, fmaf(-sn0, ab.w, acc[0].x));
                        acc[0].y = fmaf(cs0, ab.y, fmaf(sn0, ab.z, acc[0].y));
                        acc[kS - 1].x = fmaf(tn, fmaf(cs0, ab.z, -sn0 * ab.y), acc[kS - 1].x);
                        acc[kS - 1].y = fmaf(tn, fmaf(cs0, ab.w, sn0 * ab.x), acc[kS - 1].y);
                    } else {
                        // (cs + i sn)(1 + t) lp + (cs - i sn)(1 - t) lm = cs sp + i sn dm
                        const float spx = fmaf(tn, ab.z, ab.x), spy = fmaf(tn, ab.w, ab.y);
                        const float dmx = fmaf(tn, ab.x, ab.z), dmy = fmaf(tn, ab.y, ab.w);
                        acc[r].x = fmaf(cs0, spx, fmaf(-sn0, dmy, acc[r].x));
                        acc[r].y = fmaf(cs0, spy, fmaf(sn0, dmx, acc[r].y));
                    }
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < NR * kS; ++r) red[threadIdx.x][r] = acc[r];
    __syncthreads();
    for (int t = threadIdx.x; t < cnt * NR; t += blockDim.x) {
        const int qq = t % cnt, r = t / cnt;
        float2 v = red[qq][r * kS];
        for (int w = 1; w < nsl; ++w) v = cadd(v, red[w * cnt + qq][r * kS]);
        const int64_t i = e0 + qq;
        if (kRowF) {
            float2 v1 = red[qq][kS - 1];
            for (int w = 1; w < nsl; ++w) v1 = cadd(v1, red[w * cnt + qq][kS - 1]);
            const float4 rf = a.rowf[i];
            v = cadd(cmul(make_float2(rf.x, rf.y), v), cmul(make_float2(rf.z, rf.w), v1));
        }
        // (ik / 16 pi^2) v
        const float sc = a.k * 0.00633257397764611f;   // k / (16 pi^2)
        const float2 far = make_float2(-sc * v.y, sc * v.x);
        const float2 out = ynear ? cadd(ynear[r * a.n + i], far) : far;
        if (a.perm) y[r * a.n + a.perm[i]] = out;
        else y[r * a.n + i] = out;
    }
}

#define BEM_DISAGG_KERNEL(NR)                                                                                       \
    __global__ void __launch_bounds__(kDisThreads) k_disaggregate_m##NR(DisaggArgs a, const float2 *__restrict__ ynear, \
                                                                        float2 *__restrict__ y, const int *skip)     \
    {                                                                                                               \
        if (skip_now(skip)) return;                                                                                 \
        disaggregate_body<NR, false, false>(a, ynear, y);                                                           \
    }
BEM_DISAGG_KERNEL(1)
BEM_DISAGG_KERNEL(2)
BEM_DISAGG_KERNEL(4)
#undef BEM_DISAGG_KERNEL

__global__ void __launch_bounds__(kDisThreads) k_disaggregate_m1t(DisaggArgs a, const float2 *__restrict__ ynear,
                                                                  float2 *__restrict__ y, const int *skip)
{
    if (skip_now(skip)) return;
    disaggregate_body<1, false, true>(a, ynear, y);
}

// The disaggregation of the transposed product: row factor a_i + b_i (s.n_i)
// from a.rowf (see k_prep_t).
__global__ void __launch_bounds__(kDisThreads) k_disaggregate_t(DisaggArgs a, const float2 *__restrict__ ynear,
                                                                float2 *__restrict__ y, const int *skip)
{
    if (skip_now(skip)) return;
    disaggregate_body<1, true, false>(a, ynear, y);
}

__global__ void __launch_bounds__(kDisThreads) k_disaggregate_tt(DisaggArgs a, const float2 *__restrict__ ynear,
                                                                 float2 *__restrict__ y, const int *skip)
{
    if (skip_now(skip)) return;
    disaggregate_body<1, true, true>(a, ynear, y);
}

// Translation table per distinct offset X (Eq. FMMBase):
//   D_L(X, s_nu) = sum_{n=0}^{L} i^n (2n+1) h_n(k|X|) P_n(X.s_nu / |X|),
// FP64, spherical Hankel functions by upward recursion (Sec. 4.2).  The
// offsets of every far level in one launch (each block's work is a short
// serial FP64 chain, so the levels' blocks run side by side).
__global__ void k_dtable(DTableArgs a)
{
    // one block per offset X: the coefficients c_n = (2n+1) i^n h_n(k|X|)
    // depend on X only and are formed once (thread 0, upward recursion);
    // threads then take antipodal direction pairs (s, -s): with
    // P_n(-t) = (-1)^n P_n(t), the even and odd partial sums give both
    // D(X, s) = E + O and D(X, -s) = E - O.
    __shared__ double2 cn[kMaxTableL + 1];
    __shared__ double inv[kMaxTableL + 1];
    int lv = 0;
    while (lv + 1 < a.nlev && (int)blockIdx.x >= a.start[lv + 1]) ++lv;
    const DTableLevel &T = a.lev[lv];
    const int o = blockIdx.x - a.start[lv];
    const double *__restrict__ offs = T.offs;
    const double *__restrict__ dirs = T.dirs;
    const int nd = T.nd, L = T.L;
    const double k = a.k;
    float2 *__restrict__ D = T.D;
    const double X0 = offs[3 * o], X1 = offs[3 * o + 1], X2 = offs[3 * o + 2];
    const double R = sqrt(X0 * X0 + X1 * X1 + X2 * X2);
    if (threadIdx.x == 0) {
        const double x = k * R;
        double sx, cx;
        sincos(x, &sx, &cx);
        // h_0 = -i e^{ix}/x, h_1 = -e^{ix}(x + i)/x^2
        double h0r = sx / x, h0i = -cx / x;
        double h1r = -(cx * x - sx) / (x * x), h1i = -(sx * x + cx) / (x * x);
        const double ix = 1.0 / x;
        for (int n = 0; n <= L; ++n) {
            double hr, hi;
            if (n == 0) { hr = h0r; hi = h0i; }
            else if (n == 1) { hr = h1r; hi = h1i; }
            else {
                const double f = (2.0 * n - 1.0) * ix;
                hr = f * h1r - h0r;
                hi = f * h1i - h0i;
                h0r = h1r; h0i = h1i; h1r = hr; h1i = hi;
            }
            // (2n+1) i^n h_n
            const double c = 2.0 * n + 1.0;
            double ar = c * hr, ai = c * hi;
            switch (n & 3) {
                case 0: cn[n] = make_double2(ar, ai); break;
                case 1: cn[n] = make_double2(-ai, ar); break;
                case 2: cn[n] = make_double2(-ar, -ai); break;
                default: cn[n] = make_double2(ai, -ar); break;
            }
            inv[n] = 1.0 / (n + 1.0);
        }
    }
    __syncthreads();
    const double iR = 1.0 / R;
    const int h = nd / 2;
    float2 *__restrict__ Drow = D + (int64_t)o * nd;
    for (int p = threadIdx.x; p < h; p += blockDim.x) {
        const double t = (X0 * dirs[3 * p] + X1 * dirs[3 * p + 1] + X2 * dirs[3 * p + 2]) * iR;
        double p0 = 1.0, p1 = t;
        double er = cn[0].x, ei = cn[0].y, odr = 0.0, odi = 0.0;
        if (L >= 1) {
            odr = cn[1].x * t;
            odi = cn[1].y * t;
        }
        for (int n = 1; n < L; ++n) {
            // P_{n+1} = ((2n+1) t P_n - n P_{n-1}) / (n+1)
            const double p2 = ((2.0 * n + 1.0) * t * p1 - n * p0) * inv[n];
            const double2 c = cn[n + 1];
            if (n & 1) { er = fma(c.x, p2, er); ei = fma(c.y, p2, ei); }
            else { odr = fma(c.x, p2, odr); odi = fma(c.y, p2, odi); }
            p0 = p1;
            p1 = p2;
        }
        Drow[p] = make_float2((float)(er + odr), (float)(ei + odi));
        Drow[p + h] = make_float2((float)(er - odr), (float)(ei - odi));
    }
}

// ------------------------------------------------------------------ incident field
// b_i = sum_src [p_inc(x_i) - gamma dp_inc/dn(x_i)] (right-hand side of
// Eq. SystemI), gamma = i/k; FP64 phases.  Output in the internal order.
__global__ void k_rhs(const double *__restrict__ cd, const float4 *__restrict__ nrm, int64_t n, double k,
                      const SourceDev *__restrict__ src, int nsrc, float2 *__restrict__ b)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x0 = cd[3 * i], x1 = cd[3 * i + 1], x2 = cd[3 * i + 2];
    const double n0 = nrm[i].x, n1 = nrm[i].y, n2 = nrm[i].z;
    double br = 0.0, bi = 0.0;
    for (int q = 0; q < nsrc; ++q) {
        const SourceDev s = src[q];
        double pr, pi, dr, di;
        if (s.kind == 0) {
            const double ph = k * (s.v[0] * x0 + s.v[1] * x1 + s.v[2] * x2);
            double sn, cs;
            sincos(ph, &sn, &cs);
            pr = s.amp[0] * cs - s.amp[1] * sn;
            pi = s.amp[0] * sn + s.amp[1] * cs;
            const double kd = k * (s.v[0] * n0 + s.v[1] * n1 + s.v[2] * n2);
            dr = -kd * pi;              // ik (d.n) p
            di = kd * pr;
        } else {
            const double d0 = x0 - s.v[0], d1 = x1 - s.v[1], d2 = x2 - s.v[2];
            const double R = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
            double sn, cs;
            sincos(k * R, &sn, &cs);
            const double g = 1.0 / (4.0 * 3.14159265358979323846 * R);
            const double gr = g * cs, gi = g * sn;
            pr = s.amp[0] * gr - s.amp[1] * gi;
            pi = s.amp[0] * gi + s.amp[1] * gr;
            const double dn = (d0 * n0 + d1 * n1 + d2 * n2) / R;
            // p (ik - 1/R) dn
            const double fr = -dn / R, fi = k * dn;
            dr = pr * fr - pi * fi;
            di = pr * fi + pi * fr;
        }
        // p - (i/k) dp
        br += pr + di / k;
        bi += pi - dr / k;
    }
    b[i] = make_float2((float)br, (float)bi);
}

// ------------------------------------------------------------------ field evaluation
// p(x) = p_inc(x) + tau sum_j [H(x)_j p_j - G(x)_j q_j] (Eq. BIE_I, lambda =
// 1; tau = +1 at exterior points, -1 at interior points): the incident field
// of the sources at x, added to (br, bi).
__device__ void field_incident(const double *xd, float k, const SourceDev *__restrict__ src, int nsrc, double &br,
                               double &bi)
{
    for (int s = 0; s < nsrc; ++s) {
        const SourceDev S = src[s];
        double sn, cs, gr, gi;
        if (S.kind == 0) {
            sincos((double)k * (S.v[0] * xd[0] + S.v[1] * xd[1] + S.v[2] * xd[2]), &sn, &cs);
            gr = cs; gi = sn;
        } else {
            const double d0 = xd[0] - S.v[0], d1 = xd[1] - S.v[1], d2 = xd[2] - S.v[2];
            const double R = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
            sincos((double)k * R, &sn, &cs);
            gr = cs / (4.0 * 3.14159265358979323846 * R);
            gi = sn / (4.0 * 3.14159265358979323846 * R);
        }
        br += S.amp[0] * gr - S.amp[1] * gi;
        bi += S.amp[0] * gi + S.amp[1] * gr;
    }
}

// Gradient of the incident fields at x (FP64): plane wave grad p = ik d p,
// point source grad p = p (ik - 1/R) (x - x0) / R.
__device__ void incident_grad(const double *xd, float k, const SourceDev *__restrict__ src, int nsrc, double *gr,
                              double *gi)
{
    for (int s = 0; s < nsrc; ++s) {
        const SourceDev S = src[s];
        double sn, cs;
        if (S.kind == 0) {
            sincos((double)k * (S.v[0] * xd[0] + S.v[1] * xd[1] + S.v[2] * xd[2]), &sn, &cs);
            // p = A e^{i phi}; ik d p = k d (i p): i p = (-p_i, p_r)
            const double pr = S.amp[0] * cs - S.amp[1] * sn, pi = S.amp[0] * sn + S.amp[1] * cs;
            for (int a = 0; a < 3; ++a) {
                gr[a] += -(double)k * S.v[a] * pi;
                gi[a] += (double)k * S.v[a] * pr;
            }
        } else {
            const double d[3] = {xd[0] - S.v[0], xd[1] - S.v[1], xd[2] - S.v[2]};
            const double R = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
            sincos((double)k * R, &sn, &cs);
            const double g = 1.0 / (4.0 * 3.14159265358979323846 * R);
            const double pr = (S.amp[0] * cs - S.amp[1] * sn) * g, pi = (S.amp[0] * sn + S.amp[1] * cs) * g;
            // p (ik - 1/R) = (-pr/R - k pi) + i (k pr - pi/R)
            const double fr = -pr / R - (double)k * pi, fi = (double)k * pr - pi / R;
            for (int a = 0; a < 3; ++a) {
                gr[a] += fr * d[a] / R;
                gi[a] += fi * d[a] / R;
            }
        }
    }
}

// The quantity and its pair sums: the field (G and H, one complex sum) or its
// gradient (grad G and grad H, three).
template <bool kGrad> struct FieldPair;
template <> struct FieldPair<false> {
    static constexpr int kN = 1;
    GhAcc acc;
    __device__ __forceinline__ explicit FieldPair(float k) { acc = GhAcc{k, make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
    // A1 = H, A0 = G
    __device__ __forceinline__ void add(float2 *v, float2 p, float2 q) const
    {
        v[0] = cadd(v[0], csub(cmul(acc.A1, p), cmul(acc.A0, q)));
    }
};
template <> struct FieldPair<true> {
    static constexpr int kN = 3;
    GradAcc acc;
    __device__ __forceinline__ explicit FieldPair(float k)
    {
        acc.k = k;
#pragma unroll
        for (int a = 0; a < 3; ++a) acc.gG[a] = acc.gH[a] = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ void add(float2 *v, float2 p, float2 q) const
    {
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = cadd(v[a], csub(cmul(acc.gH[a], p), cmul(acc.gG[a], q)));
    }
};
// The contribution of element j at x by the general element rules.
template <bool kGrad>
__device__ __noinline__ bool field_entry(const ElemDev &E, const QuadTables &Q, int64_t j, const double *xd, float k,
                                         float2 p, float2 q, float2 *v)
{
    const float3 xhi = make_float3((float)xd[0], (float)xd[1], (float)xd[2]);
    const float3 xlo = make_float3((float)(xd[0] - (double)xhi.x), (float)(xd[1] - (double)xhi.y),
                                   (float)(xd[2] - (double)xhi.z));
    FieldPair<kGrad> f(k);
    const bool ok = integrate_regular_acc(E, j, xhi, xlo, xd, Q, f.acc);
    for (int a = 0; a < FieldPair<kGrad>::kN; ++a) v[a] = make_float2(0.f, 0.f);
    f.add(v, p, q);
    return ok;
}

// x_j - x of element j and a point x.
__device__ __forceinline__ float3 point_to(const ElemDev &E, int64_t j, const double *xd)
{
    const float3 xhi = make_float3((float)xd[0], (float)xd[1], (float)xd[2]);
    const float3 xlo = make_float3((float)(xd[0] - (double)xhi.x), (float)(xd[1] - (double)xhi.y),
                                   (float)(xd[2] - (double)xhi.z));
    return add3(sub3f(f3(E.chi[j]), xhi), sub3f(f3(E.clo[j]), xlo));
}
__device__ __noinline__ int cut_point(const ElemDev &E, const QuadTables &Q, int64_t j, const double *xd, unsigned *out,
                                      int cap)
{
    return cut_element(E, Q, j, point_to(E, j, xd), xd, out, cap);
}
// The contribution of a part of element j at x.
template <bool kGrad>
__device__ __forceinline__ void field_part(const ElemDev &E, int64_t j, const double *xd, unsigned code,
                                           const float4 *rule, float k, float2 p, float2 q, float2 *v)
{
    const int m = (code >> 24) & 7, depth = (code >> 20) & 15;
    const SubTri T = part_triangle(code, depth);
    const float3 g1 = f3(E.e1[j]), g2 = f3(E.e2[j]), ny = f3(E.nrm[j]);
    const float3 base = add3(point_to(E, j, xd), f3(E.va[j]));
    const float sa = E.chi[j].w * exp2f(-2.0f * (float)depth);
    const float sx1 = T.x1 - T.x0, sy1 = T.y1 - T.y0, sx2 = T.x2 - T.x0, sy2 = T.y2 - T.y0;
    FieldPair<kGrad> f(k);
    const int r1 = rule_at(m + 1);
    for (int u = rule_at(m); u < r1; ++u) {
        const float4 rl = rule[u];
        const float px = T.x0 + rl.x * sx1 + rl.y * sx2, py = T.y0 + rl.x * sy1 + rl.y * sy2;
        f.acc.point(mad3(py, g2, mad3(px, g1, base)), ny, sa * rl.z);
    }
#pragma unroll
    for (int a = 0; a < FieldPair<kGrad>::kN; ++a) v[a] = make_float2(0.f, 0.f);
    f.add(v, p, q);
}

// Direct sum over every element at M points: p (k_field) or v (k_field_
// velocity).  Bound by FP32 / SFU issue.  As in the recomputed product, a lane
// holds a point, the elements are staged in shared memory in tiles of `cols`
// and read as broadcasts (their vertices, which order 1 does not need, from
// global memory: staged, far points took 4 % longer and points at the surface 3 %
// less), and the pairs under one rule of order 1 to 3 are evaluated in place; the
// others (subdivided elements, orders 4 to 6, distances
// within rounding of a threshold) are queued per block and worked off as there
// (work_queue), their sums FP64 additions.  Block (x, y) takes `rows` points and every gridDim.y-th part of
// the elements; with several parts they go to part[(m S + s) N + a] and the
// finish kernels add them in order.  rows, cols and the parts are
// fused_split's: few points or few elements get small blocks.
// Calls (host part of about 60 us included) on 5120 elements: 3000 points 0.2 m
// off the surface 139 us, a millimetre off it 345; with one point per block and
// lanes over the elements (112 bytes of element data through L1 per pair) 232
// and 915.  200 points at a surface of 320 elements 130 and 186 us; with orders
// 2 and 3 queued as well, and pairs worked off whole, one per thread, 1758.
template <bool kGrad>
__device__ __forceinline__ void field_body(const ElemDev &E, const QuadTables &Q, const double *__restrict__ pts,
                                           int64_t M, int rows, int cols, float k, float tau, float inv_omega_rho,
                                           const float2 *__restrict__ p, const float2 *__restrict__ qs,
                                           const SourceDev *__restrict__ src, int nsrc, float2 *__restrict__ part,
                                           float2 *__restrict__ out, int *err)
{
    constexpr int kW = kFusedThreads / 32, kN = FieldPair<kGrad>::kN;
    // the staged tile, and afterwards the parts of the queued pairs
    constexpr int kTileBytes = 4 * kFusedTile * 16;
    __shared__ __align__(16) unsigned char s_buf[kTileBytes > 10 * kFieldParts ? kTileBytes : 10 * kFieldParts];
    float4 *s_hi = reinterpret_cast<float4 *>(s_buf), *s_lo = s_hi + kFusedTile, *s_n = s_lo + kFusedTile;
    float4 *s_pq = s_n + kFusedTile;
    __shared__ float4 s_rule[91];                      // (xi, eta, 2 w) of orders 1 to 6
    __shared__ int s_pn[8];
    __shared__ int s_qj[kFieldQueue];
    __shared__ unsigned char s_qr[kFieldQueue];
    __shared__ int s_qn;
    __shared__ double2 s_h[kN][32];
    __shared__ double s_x[32][3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t m0 = (int64_t)blockIdx.x * rows;
    const int cnt = (int)min((int64_t)rows, M - m0);
    int w = 1;
    while (w < cnt) w <<= 1;
    const int R = 32 / w, sub = lane / w, rr = lane % w;   // R elements side by side for w < 32 points
    const bool live = rr < cnt;
    if (threadIdx.x < 32) {
#pragma unroll
        for (int a = 0; a < kN; ++a) s_h[a][threadIdx.x] = make_double2(0.0, 0.0);
        for (int a = 0; a < 3; ++a) s_x[threadIdx.x][a] = (int)threadIdx.x < cnt ? pts[3 * (m0 + threadIdx.x) + a] : 0.0;
    }
    if (threadIdx.x < 91) s_rule[threadIdx.x] = rule_point(Q, threadIdx.x);
    if (threadIdx.x == 0) s_qn = 0;
    __syncthreads();
    const double *xd = s_x[live ? rr : 0];
    const float3 xhi = make_float3((float)xd[0], (float)xd[1], (float)xd[2]);
    const float3 xlo = make_float3((float)(xd[0] - (double)xhi.x), (float)(xd[1] - (double)xhi.y),
                                   (float)(xd[2] - (double)xhi.z));
    // thresholds on r~^2 as in the recomputed product
    const float rt1 = fmaxf(Q.R2[1] * (1.0f + 2e-5f), Q.whole_rt2);
    const float rt1lo = Q.R2[1] * (1.0f - 2e-5f), rt2hi = Q.R2[2] * (1.0f + 2e-5f), rt2lo = Q.R2[2] * (1.0f - 2e-5f);
    const float rth = Q.m_max > 3 ? Q.heavy_rt2 : Q.whole_rt2;
    // the queued pairs (called by the whole block after a barrier; takes the
    // staged tile's place)
    auto drain = [&]() {
        auto add = [&](int row, const float2 *v) {
#pragma unroll
            for (int a = 0; a < kN; ++a) {
                atomicAdd(&s_h[a][row].x, (double)v[a].x);
                atomicAdd(&s_h[a][row].y, (double)v[a].y);
            }
        };
        work_queue<kFusedThreads, kFieldParts>(
            min(s_qn, kFieldQueue), s_buf, s_pn,
            [&](int q, unsigned *out, int cap) { return cut_point(E, Q, s_qj[q], s_x[s_qr[q]], out, cap); },
            [&](int q, unsigned code) {
                float2 v[kN];
                field_part<kGrad>(E, s_qj[q], s_x[s_qr[q]], code, s_rule, k, p[s_qj[q]], qs[s_qj[q]], v);
                add(s_qr[q], v);
            },
            [&](int q) {                               // cut deeper than a code can say
                float2 v[kN];
                if (field_entry<kGrad>(E, Q, s_qj[q], s_x[s_qr[q]], k, p[s_qj[q]], qs[s_qj[q]], v)) add(s_qr[q], v);
                else atomicMin(err, s_qj[q]);
            });
        if (threadIdx.x == 0) s_qn = 0;
    };
    float2 acc[kN];
#pragma unroll
    for (int a = 0; a < kN; ++a) acc[a] = make_float2(0.f, 0.f);
    const int S = gridDim.y, sl = blockIdx.y, chunk = cols / kW;
    const int64_t ntile = (E.n + cols - 1) / cols;
    const int64_t tb = ntile * sl / S, te = ntile * (sl + 1) / S;
    unsigned pend = 0;                                 // elements of this lane that found the queue full
    for (int64_t tile = tb;; ++tile) {
        // as in the recomputed product (s_qn is the same in every thread: no
        // pushes since the barrier)
        for (;;) {
            const bool full = __syncthreads_or(pend != 0);
            if (!full && (tile < te ? s_qn <= kFieldQueue / 2 : s_qn == 0)) break;
            drain();
            __syncthreads();
            if (!full) break;
            for (unsigned left = pend; left; left &= left - 1) {
                const int b = __ffs((int)left) - 1, slot = atomicAdd(&s_qn, 1);
                if (slot >= kFieldQueue) break;
                s_qj[slot] = (int)((tile - 1) * cols) + warp * chunk + b;
                s_qr[slot] = (unsigned char)rr;
                pend &= ~(1u << b);
            }
        }
        if (tile >= te) break;
        const int64_t j = tile * cols + threadIdx.x;
        if ((int)threadIdx.x < cols && j < E.n) {
            const float4 h = E.chi[j];
            float4 l = E.clo[j];
            l.w = __frcp_rn(h.w);
            const float2 pj = p[j], qj = qs[j];
            s_hi[threadIdx.x] = h;
            s_lo[threadIdx.x] = l;
            s_n[threadIdx.x] = E.nrm[j];
            s_pq[threadIdx.x] = make_float4(pj.x, pj.y, qj.x, qj.y);
        }
        __syncthreads();
        const int c0 = warp * chunk, c1 = (int)min((int64_t)c0 + chunk, E.n - tile * cols);
        float2 ta[kN];                                      // the tile's own sum first
#pragma unroll
        for (int a = 0; a < kN; ++a) ta[a] = make_float2(0.f, 0.f);
        for (int cb = c0; cb < c1; cb += R) {
            const int c = cb + sub;
            if (!live || c >= c1) continue;
            const float4 eh = s_hi[c], el = s_lo[c];
            float3 D0;
            const float rt2 = pair_rt2(f3(eh), f3(el), xhi, xlo, el.w, D0);
            int code = 0;
            if (rt2 > rt1) code = 1;
            else if (rt2 > rth && rt2 < rt1lo && (rt2 > rt2hi || rt2 < rt2lo)) code = rt2 > rt2hi ? 2 : 3;
            if (code == 0) {
                const int slot = atomicAdd(&s_qn, 1);
                if (slot < kFieldQueue) {
                    s_qj[slot] = (int)(tile * cols) + c;
                    s_qr[slot] = (unsigned char)rr;
                } else {
                    pend |= 1u << (c - c0);
                }
                continue;
            }
            const float4 pq = s_pq[c];
            const float3 ny = f3(s_n[c]);
            FieldPair<kGrad> f(k);
            if (code == 1) {
                f.acc.point(D0, ny, eh.w);
            } else {
                const int64_t je = tile * cols + c;
                const float3 g1 = f3(E.e1[je]), g2 = f3(E.e2[je]), base = add3(D0, f3(E.va[je]));
                const int u1 = code == 2 ? 5 : 14;
                for (int u = code == 2 ? 1 : 5; u < u1; ++u) {
                    const float4 rl = s_rule[u];
                    f.acc.point(mad3(rl.y, g2, mad3(rl.x, g1, base)), ny, eh.w * rl.z);
                }
            }
            f.add(ta, make_float2(pq.x, pq.y), make_float2(pq.z, pq.w));
        }
#pragma unroll
        for (int a = 0; a < kN; ++a) acc[a] = cadd(acc[a], ta[a]);
    }
    // the sums of a point: elements side by side in a warp, then the warps in order
    float2 *red = reinterpret_cast<float2 *>(s_hi);
    float2 tot[kN];
#pragma unroll
    for (int a = 0; a < kN; ++a) {
        __syncthreads();
        red[threadIdx.x] = lanes_sum(acc[a], w);
        __syncthreads();
        if ((int)threadIdx.x < cnt) {
            Sum2 v(s_h[a][threadIdx.x]);
            for (int u = 0; u < kW; ++u) v.add(red[u * 32 + threadIdx.x]);
            tot[a] = cscale(v.value(), tau);                // tau on the integral part (Eq. BIE_I)
        }
    }
    if ((int)threadIdx.x >= cnt) return;
    const int64_t m = m0 + threadIdx.x;
    if (S > 1) {
#pragma unroll
        for (int a = 0; a < kN; ++a) part[(m * S + sl) * kN + a] = tot[a];
    } else if (!kGrad) {
        double br = tot[0].x, bi = tot[0].y;
        field_incident(s_x[threadIdx.x], k, src, nsrc, br, bi);
        out[m] = make_float2((float)br, (float)bi);
    } else {
        double gr[3], gi[3];
#pragma unroll
        for (int a = 0; a < kN; ++a) {
            gr[a] = tot[a].x;
            gi[a] = tot[a].y;
        }
        incident_grad(s_x[threadIdx.x], k, src, nsrc, gr, gi);
        // v = grad p / (i w rho) = -i grad p / (w rho)
        for (int a = 0; a < kN; ++a)
            out[3 * m + a] = make_float2((float)(gi[a] * inv_omega_rho), (float)(-gr[a] * inv_omega_rho));
    }
}

__global__ void __launch_bounds__(kFusedThreads, 3) k_field(ElemDev E, const QuadTables *__restrict__ Q,
                                                         const double *__restrict__ pts, int64_t M, int rows, int cols,
                                                         float k, float tau, const float2 *__restrict__ p, const float2 *__restrict__ q,
                                                         const SourceDev *__restrict__ src, int nsrc,
                                                         float2 *__restrict__ part, float2 *__restrict__ out, int *err)
{
    field_body<false>(E, *Q, pts, M, rows, cols, k, tau, 0.f, p, q, src, nsrc, part, out, err);
}

// Particle velocity at field points, v = grad p / (i w rho) (Eq. utopandv),
// with grad p = grad p_inc + tau sum_j [grad H(x)_j p_j - grad G(x)_j q_j]
// (Eq. BIE_I, lambda = 1, differentiated under the integral; the element
// rules of the field).  out: [M][3] (x, y, z components).
__global__ void __launch_bounds__(kFusedThreads, 3) k_field_velocity(ElemDev E, const QuadTables *__restrict__ Q,
                                                                  const double *__restrict__ pts, int64_t M, int rows,
                                                                  int cols, float k, float tau, float inv_omega_rho,
                                                                  const float2 *__restrict__ p,
                                                                  const float2 *__restrict__ q,
                                                                  const SourceDev *__restrict__ src, int nsrc,
                                                                  float2 *__restrict__ part, float2 *__restrict__ out,
                                                                  int *err)
{
    field_body<true>(E, *Q, pts, M, rows, cols, k, tau, inv_omega_rho, p, q, src, nsrc, part, out, err);
}

// The S partial sums of a point, `stride` apart, by one thread, or by a warp
// (every lane takes part; the lanes are added in a fixed tree).
__device__ __forceinline__ double2 finish_sum(const float2 *__restrict__ part, int stride, int S, int lanes)
{
    Sum2 v;
#pragma unroll 4
    for (int s = threadIdx.x % lanes; s < S; s += lanes) v.add(part[s * stride]);
    if (lanes > 1)
        for (int o = 16; o > 0; o >>= 1) {
            const float2 t = make_float2(__shfl_xor_sync(0xffffffffu, v.s.x, o), __shfl_xor_sync(0xffffffffu, v.s.y, o));
            const float2 u = make_float2(__shfl_xor_sync(0xffffffffu, v.e.x, o), __shfl_xor_sync(0xffffffffu, v.e.y, o));
            v.add(t);
            v.e = cadd(v.e, u);
        }
    return v.value_d();
}

// The S partial sums of each field point, plus the incident field.
__global__ void k_field_finish(const double *__restrict__ pts, int64_t M, int S, int lanes, float k,
                               const SourceDev *__restrict__ src, int nsrc, const float2 *__restrict__ part,
                               float2 *__restrict__ out)
{
    const int64_t m = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / lanes;
    if (m >= M) return;
    const double2 v = finish_sum(part + m * S, 1, S, lanes);
    if (threadIdx.x % lanes > 0) return;
    const double xd[3] = {pts[3 * m], pts[3 * m + 1], pts[3 * m + 2]};
    double br = v.x, bi = v.y;
    field_incident(xd, k, src, nsrc, br, bi);
    out[m] = make_float2((float)br, (float)bi);
}

// Far-field weights of the representation formula (Eq. BIE with lambda = 1)
// for the aggregation T(l) (Sec. 3.3.3): with the one-point element rule,
//   H_j p_j - G_j q_j ~ A_j (-q_j - ik (n_j.s) p_j) e^{ik (z_s - y_j).s} (...),
// i.e. (alpha, c) = (-A q, -ik A p) in the form sum_j E_pj (alpha_j + t_pj c_j)
// of the aggregation (internal element order).
__global__ void k_field_weights(int64_t n, const float2 *__restrict__ p, const float2 *__restrict__ q,
                                const float4 *__restrict__ chi, float k, float4 *__restrict__ wts)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float A = chi[i].w;
    const float2 pv = p[i], qv = q[i];
    wts[i] = make_float4(-A * qv.x, -A * qv.y, k * A * pv.y, -k * A * pv.x);
}

// Rule of the pair of a point and an element: 1 to 3 where one regular rule of
// that order serves the whole element, else 0, an expensive pair (thresholds on
// r~^2 as in the recomputed product; FP64 within rounding of R_1 and R_2).
__device__ __forceinline__ int light_rule(const ElemDev &E, const QuadTables &Q, int j, float3 D0, float area, float rt2,
                                          const double *xd)
{
    if (rt2 > fmaxf(Q.R2[1] * (1.0f + 2e-5f), Q.whole_rt2)) return 1;
    if (!(rt2 > (Q.m_max > 3 ? Q.heavy_rt2 : Q.whole_rt2))) return 0;
    if (rt2 < Q.R2[1] * (1.0f - 2e-5f)) {
        if (rt2 > Q.R2[2] * (1.0f + 2e-5f)) return 2;
        if (rt2 < Q.R2[2] * (1.0f - 2e-5f)) return 3;
    }
    const int code = whole_rule(E, j, D0, area, xd, Q);
    return code <= 3 ? code : 0;
}
// Near part of the field at points (internal point order): the element rules
// of the direct sum over the point's leaf near list, kFieldNearWarps warps per
// point; v_m = sum_j H_j p_j - G_j q_j.  The list's runs (first element, first
// position) are walked by position, so that all lanes have an element whatever
// the runs' lengths (a run is often a leaf of a dozen elements).  The pairs of
// orders 1 to 3 here, with few registers and one barrier, since most points have
// no others; the points close to the surface are listed in close (their number
// first) for k_field_near_close.  24,874 points around 20,480 elements: 35 us, and
// 6 for the empty second launch (all rules in one kernel, 92 registers: 43; one
// warp per point 74).
__global__ void __launch_bounds__(32 * kFieldNearWarps)
k_field_near(ElemDev E, const QuadTables *__restrict__ Qp, const double *__restrict__ pts, float k,
             const float2 *__restrict__ p, const float2 *__restrict__ q, const int *__restrict__ pleaf,
             const int *__restrict__ nptr, const int *__restrict__ ntot, const int2 *__restrict__ nruns,
             float2 *__restrict__ v, int *__restrict__ close)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t m = blockIdx.x;
    const int pl = pleaf[m], tot = ntot[pl], r1 = nptr[pl + 1];
    if (tot == 0) {                                    // far from every element
        if (threadIdx.x == 0) v[m] = make_float2(0.f, 0.f);
        return;
    }
    float2 acc = make_float2(0.f, 0.f);
    bool expensive = false;
    if ((int)threadIdx.x < tot) {                      // (the point's FP64 conversions are most of a short list)
        const QuadTables &Q = *Qp;
        const double xd[3] = {pts[3 * m], pts[3 * m + 1], pts[3 * m + 2]};
        const float3 xhi = make_float3((float)xd[0], (float)xd[1], (float)xd[2]);
        const float3 xlo = make_float3((float)(xd[0] - (double)xhi.x), (float)(xd[1] - (double)xhi.y),
                                       (float)(xd[2] - (double)xhi.z));
        int r = nptr[pl];
        for (int c = threadIdx.x; c < tot; c += 32 * kFieldNearWarps) {
            while (r + 1 < r1 && nruns[r + 1].y <= c) ++r;
            const int2 run = nruns[r];
            const int j = run.x + (c - run.y);
            const float4 h = E.chi[j];
            const float3 ny = f3(E.nrm[j]);
            float3 D0;
            const float rt2 = pair_rt2(f3(h), f3(E.clo[j]), xhi, xlo, __frcp_rn(h.w), D0);
            const int code = light_rule(E, Q, j, D0, h.w, rt2, xd);
            FieldPair<false> f(k);
            if (code == 1) {
                f.acc.point(D0, ny, h.w);
            } else if (code > 1) {
                const float3 g1 = f3(E.e1[j]), g2 = f3(E.e2[j]), base = add3(D0, f3(E.va[j]));
                for (int u = 0; u < code * code; ++u)
                    f.acc.point(mad3(Q.tri_eta[code][u], g2, mad3(Q.tri_xi[code][u], g1, base)), ny,
                                2.0f * h.w * Q.tri_w[code][u]);
            } else {
                expensive = true;
            }
            f.add(&acc, p[j], q[j]);
        }
    }
    __shared__ float2 red[kFieldNearWarps];
    acc = warp_sum(acc);
    if (lane == 0) red[warp] = acc;
    const bool any = __syncthreads_or(expensive);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < kFieldNearWarps; ++w) acc = cadd(acc, red[w]);
        v[m] = acc;
        if (any) close[1 + atomicAdd(close, 1)] = (int)m;
    }
}

// The expensive pairs of the listed points, added to v: a block goes over a
// point's list again, queues them and works them off part by part (work_queue).
// 5000 points a millimetre off 1280 elements: 630 us a call (lanes that took such
// a pair whole, as the general rule does: 957).
__global__ void __launch_bounds__(32 * kFieldNearWarps, 5)
k_field_near_close(ElemDev E, const QuadTables *__restrict__ Qp, const double *__restrict__ pts, float k,
                   const float2 *__restrict__ p, const float2 *__restrict__ q, const int *__restrict__ pleaf,
                   const int *__restrict__ nptr, const int *__restrict__ ntot, const int2 *__restrict__ nruns,
                   float2 *__restrict__ v, const int *__restrict__ close, int *err)
{
    constexpr int kT = 32 * kFieldNearWarps;
    static_assert(kFieldNearQueue >= 4 * kT, "two passes of pushes find room above the half");
    __shared__ __align__(16) unsigned char s_buf[10 * kFieldNearParts];
    __shared__ float4 s_rule[91];                      // (xi, eta, 2 w) of orders 1 to 6
    __shared__ int s_qj[kFieldNearQueue], s_qn, s_pn[8];
    __shared__ double s_x[3];
    __shared__ double2 s_h;
    const QuadTables &Q = *Qp;
    const int n = *close;
    if (blockIdx.x >= n) return;
    if (threadIdx.x < 91) s_rule[threadIdx.x] = rule_point(Q, threadIdx.x);
    auto add = [&](float2 u) {
        atomicAdd(&s_h.x, (double)u.x);
        atomicAdd(&s_h.y, (double)u.y);
    };
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        const int m = close[1 + i];
        __syncthreads();                               // the point before has been written
        if (threadIdx.x < 3) s_x[threadIdx.x] = pts[3 * (int64_t)m + threadIdx.x];
        if (threadIdx.x == 0) {
            s_qn = 0;
            s_h = make_double2(0.0, 0.0);
        }
        __syncthreads();
        const int pl = pleaf[m], tot = ntot[pl], r1 = nptr[pl + 1];
        const float3 xhi = make_float3((float)s_x[0], (float)s_x[1], (float)s_x[2]);
        const float3 xlo = make_float3((float)(s_x[0] - (double)xhi.x), (float)(s_x[1] - (double)xhi.y),
                                       (float)(s_x[2] - (double)xhi.z));
        int r = nptr[pl];
        bool half = false;                             // this thread queued a pair beyond half of the queue
        for (int c0 = 0, pass = 1; c0 < tot; c0 += kT, ++pass) {
            const int c = c0 + threadIdx.x;
            if (c < tot) {
                while (r + 1 < r1 && nruns[r + 1].y <= c) ++r;
                const int2 run = nruns[r];
                const int j = run.x + (c - run.y);
                const float4 h = E.chi[j];
                float3 D0;
                const float rt2 = pair_rt2(f3(h), f3(E.clo[j]), xhi, xlo, __frcp_rn(h.w), D0);
                if (light_rule(E, Q, j, D0, h.w, rt2, s_x) == 0) {
                    const int slot = atomicAdd(&s_qn, 1);
                    s_qj[slot] = j;
                    half = half || slot >= kFieldNearQueue / 2;
                }
            }
            // a barrier every second pass
            const bool last = c0 + kT >= tot;
            if (!last && (pass & 1)) continue;
            if (!__syncthreads_or(half) && !last) continue;
            work_queue<kT, kFieldNearParts>(
                s_qn, s_buf, s_pn, [&](int u, unsigned *out, int cap) { return cut_point(E, Q, s_qj[u], s_x, out, cap); },
                [&](int u, unsigned code) {
                    float2 w;
                    field_part<false>(E, s_qj[u], s_x, code, s_rule, k, p[s_qj[u]], q[s_qj[u]], &w);
                    add(w);
                },
                [&](int u) {                           // cut deeper than a code can say
                    float2 w;
                    if (field_entry<false>(E, Q, s_qj[u], s_x, k, p[s_qj[u]], q[s_qj[u]], &w)) add(w);
                    else atomicMin(err, s_qj[u]);
                });
            if (threadIdx.x == 0) s_qn = 0;
            half = false;
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            Sum2 t(s_h);
            t.add(v[m]);
            v[m] = t.value();
        }
    }
}

// The field at the points: tau (near + far) plus the incident field (FP64),
// written in caller order.
__global__ void k_field_eval_finish(const double *__restrict__ pts, int64_t M, float k, float tau,
                                    const SourceDev *__restrict__ src, int nsrc, const float2 *__restrict__ v,
                                    const int64_t *__restrict__ perm, float2 *__restrict__ out)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const double xd[3] = {pts[3 * m], pts[3 * m + 1], pts[3 * m + 2]};
    const float2 w = cscale(v[m], tau);
    double br = w.x, bi = w.y;
    field_incident(xd, k, src, nsrc, br, bi);
    out[perm[m]] = make_float2((float)br, (float)bi);
}

// The S partial gradients of each field point, the incident gradient and the
// scaling to the velocity.
__global__ void k_field_velocity_finish(const double *__restrict__ pts, int64_t M, int S, int lanes, float k,
                                        float inv_omega_rho, const SourceDev *__restrict__ src, int nsrc,
                                        const float2 *__restrict__ part, float2 *__restrict__ out)
{
    const int64_t m = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / lanes;
    if (m >= M) return;
    double gr[3], gi[3];
    for (int a = 0; a < 3; ++a) {
        const double2 v = finish_sum(part + m * S * 3 + a, 3, S, lanes);
        gr[a] = v.x;
        gi[a] = v.y;
    }
    if (threadIdx.x % lanes > 0) return;
    const double xd[3] = {pts[3 * m], pts[3 * m + 1], pts[3 * m + 2]};
    incident_grad(xd, k, src, nsrc, gr, gi);
    for (int a = 0; a < 3; ++a)
        out[3 * m + a] = make_float2((float)(gi[a] * inv_omega_rho), (float)(-gr[a] * inv_omega_rho));
}

// ------------------------------------------------------------------ vector helpers
__global__ void k_gather(const float2 *__restrict__ x, const int64_t *__restrict__ perm, int64_t n,
                         float2 *__restrict__ y)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = x[perm[i]];
}
__global__ void k_gather2(const float2 *__restrict__ x0, const float2 *__restrict__ x1,
                          const int64_t *__restrict__ perm, int64_t n, float2 *__restrict__ y0, float2 *__restrict__ y1)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t j = perm[i];
    y0[i] = x0[j];
    y1[i] = x1[j];
}
// The boundary conditions folded into column coefficients (Eq. SystemI):
// column j enters as p_j = cp u_j, q_j = cq u_j, with (1, 0) for VELO, (1, a)
// for ADMI, a = -tau i k rho c Y (Y = velocity into the wall / p; the wall lies
// along the normal for the interior problem, against it for the exterior
// one), and (0, 1) for PRES; (cp0, cq0) and z the same for the known data
// g = i w rho v and p.  tau multiplies every integral operator, so all but
// aq and z carry it.  Formed here from the boundary data on the device: on
// the host, the six vectors, their uploads and a comparison with the last
// call's took 0.17 ms of every product on 20,480 elements and 2.9 ms on
// 158,420; this takes one launch when something changed.
__global__ void k_coeffs(int64_t n, const int *__restrict__ type, const double2 *__restrict__ bcv,
                         const int *__restrict__ region, const double *__restrict__ adm, double k, double omega,
                         double rho, double c, double tau, float2 *__restrict__ cp, float2 *__restrict__ cq,
                         float2 *__restrict__ cp0, float2 *__restrict__ cq0, float2 *__restrict__ z,
                         float2 *__restrict__ aq)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int ty = type[i];
    const double2 v = bcv[i];
    const float2 one = make_float2(1.f, 0.f), zero = make_float2(0.f, 0.f);
    float2 p = zero, q = zero, p0 = zero, q0 = zero, zz, a = zero;
    if (ty == BEM_PRES) {
        q = p0 = one;
        zz = make_float2((float)v.x, (float)v.y);
    } else {
        p = q0 = one;
        zz = make_float2((float)(-omega * rho * v.y), (float)(omega * rho * v.x));
        if (ty == BEM_ADMI) {
            const int r = region[i];
            const double br = tau * rho * c * adm[2 * r], bi = tau * rho * c * adm[2 * r + 1];
            q = a = make_float2((float)(k * bi), (float)(-k * br));
        }
    }
    z[i] = zz;
    aq[i] = a;
    if (tau < 0) {
        p = make_float2(-p.x, -p.y);
        q = make_float2(-q.x, -q.y);
        p0 = make_float2(-p0.x, -p0.y);
        q0 = make_float2(-q0.x, -q0.y);
    }
    cp[i] = p;
    cq[i] = q;
    cp0[i] = p0;
    cq0[i] = q0;
}
// Iterative refinement of a mixed-precision solve: r = b - y in FP64 from the
// FP32 right-hand side and product (y = A x with the FP32 products), stored
// as FP32 in r; part[blockIdx.x] = the block's ||r||^2 in FP64.
__global__ void k_refine_residual(const float2 *__restrict__ b, const float2 *__restrict__ y, float2 *__restrict__ r,
                                  int64_t n, double *__restrict__ part)
{
    double v = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double rx = (double)b[i].x - (double)y[i].x, ry = (double)b[i].y - (double)y[i].y;
        r[i] = make_float2((float)rx, (float)ry);
        v += rx * rx + ry * ry;
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __shared__ double red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) part[blockIdx.x] = s;
    }
}

// x64 += d (the refinement's FP64 solution) and x = x64 rounded to FP32.
__global__ void k_refine_update(double2 *__restrict__ x64, const float2 *__restrict__ d, float2 *__restrict__ x,
                                int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 v = make_double2(x64[i].x + (double)d[i].x, x64[i].y + (double)d[i].y);
    x64[i] = v;
    x[i] = make_float2((float)v.x, (float)v.y);
}

// b <- b - y
__global__ void k_sub(float2 *__restrict__ b, const float2 *__restrict__ y, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = csub(b[i], y[i]);
}
// w <- b - w
__global__ void k_rsub(float2 *__restrict__ w, const float2 *__restrict__ b, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) w[i] = csub(b[i], w[i]);
}
// p, q from the unknowns u and the known data z (internal order), written in
// the caller order: VELO/ADMI: p = u, q = a u + z; PRES: p = z, q = u.
__global__ void k_pq(const float2 *__restrict__ u, const float2 *__restrict__ z, const float2 *__restrict__ aq,
                     const int *__restrict__ type, const int64_t *__restrict__ perm, int64_t n,
                     float2 *__restrict__ p, float2 *__restrict__ q)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float2 pv, qv;
    if (type[i] == 1) { pv = z[i]; qv = u[i]; }
    else { pv = u[i]; qv = cfma(aq[i], u[i], z[i]); }
    p[perm[i]] = pv;
    if (q) q[perm[i]] = qv;
}


// ------------------------------------------------------------------ GMRES
// Givens step (FP64), run by one warp: h_{j+1,j} = ||w|| (nn = ||w||^2),
// apply the previous rotations to column j, form the new rotation, update g
// and the residual estimate, and decide whether the cycle ends.
//
// Rotation l maps (t_l, h_{l+1}) to (conj(c_l) t_l + s_l h_{l+1},
// -s_l t_l + c_l h_{l+1}) with s_l real, so the running entry obeys the affine
// recurrence t_{l+1} = a_l t_l + b_l, a_l = -s_l, b_l = c_l h_{l+1}.  The warp
// composes these maps with a prefix scan (|a_l| <= 1: no growth) instead of
// applying j rotations one after another in one thread: FP64 issue is scarce
// on this part, and the serial chain costs j times its latency.
__device__ void gm_givens_warp(const GmresArgs &a, double nn, int j)
{
    __shared__ double2 sh[kMaxRestart + 1], shr[kMaxRestart + 1];
    __shared__ double2 s_tj;
    GmresState *st = a.st;
    const int m = a.m;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    for (int l = lane; l <= j; l += 32) sh[l] = __ldcg(a.H + (int64_t)l * m + j);
    __syncwarp();
    const int K = (j + 31) / 32;                 // rotations per lane
    const int l0 = min(j, lane * K), l1 = min(j, l0 + K);
    double A = 1.0;
    double2 B = make_double2(0.0, 0.0);
    for (int l = l0; l < l1; ++l) {
        const double2 c = __ldcg(a.cs + l);
        const double sl = __ldcg(&a.sn[l].x);
        const double2 h1 = sh[l + 1];
        const double bx = c.x * h1.x - c.y * h1.y, by = c.x * h1.y + c.y * h1.x;
        A = -sl * A;
        B = make_double2(fma(-sl, B.x, bx), fma(-sl, B.y, by));
    }
    // inclusive scan: mine o (lane - o)'s
    for (int o = 1; o < 32; o <<= 1) {
        const double Ap = __shfl_up_sync(full, A, o);
        const double Bx = __shfl_up_sync(full, B.x, o), By = __shfl_up_sync(full, B.y, o);
        if (lane >= o) {
            B = make_double2(fma(A, Bx, B.x), fma(A, By, B.y));
            A *= Ap;
        }
    }
    double Ae = __shfl_up_sync(full, A, 1);
    double Bex = __shfl_up_sync(full, B.x, 1), Bey = __shfl_up_sync(full, B.y, 1);
    if (lane == 0) { Ae = 1.0; Bex = 0.0; Bey = 0.0; }
    const double2 h0 = sh[0];
    double2 t = make_double2(fma(Ae, h0.x, Bex), fma(Ae, h0.y, Bey));
    for (int l = l0; l < l1; ++l) {
        const double2 c = __ldcg(a.cs + l);
        const double sl = __ldcg(&a.sn[l].x);
        const double2 h1 = sh[l + 1];
        shr[l] = make_double2(c.x * t.x + c.y * t.y + sl * h1.x, c.x * t.y - c.y * t.x + sl * h1.y);
        t = make_double2(-sl * t.x + c.x * h1.x - c.y * h1.y, -sl * t.y + c.x * h1.y + c.y * h1.x);
    }
    if ((j == 0 && lane == 0) || (l0 < l1 && l1 == j)) s_tj = t;
    __syncwarp();
    if (lane == 0) {
        const double hn = sqrt(nn);
        const double2 hj = s_tj;
        const double den = sqrt(hj.x * hj.x + hj.y * hj.y + hn * hn);
        double2 c, sv;
        if (den == 0.0) { c = make_double2(1.0, 0.0); sv = make_double2(0.0, 0.0); }
        else { c = make_double2(hj.x / den, hj.y / den); sv = make_double2(hn / den, 0.0); }
        a.cs[j] = c;
        a.sn[j] = sv;
        shr[j] = make_double2(den, 0.0);
        shr[j + 1] = make_double2(0.0, 0.0);
        const double2 g0 = a.g[j];
        a.g[j] = make_double2(c.x * g0.x + c.y * g0.y, c.x * g0.y - c.y * g0.x);
        const double2 g1 = make_double2(-(sv.x * g0.x - sv.y * g0.y), -(sv.x * g0.y + sv.y * g0.x));
        a.g[j + 1] = g1;
        const double res = sqrt(g1.x * g1.x + g1.y * g1.y) / st->bnorm;
        st->resid = res;
        st->iters += 1;
        st->hn = hn;
        st->ncols = j + 1;
        if (res <= st->tol || hn <= 1e-300 * st->bnorm || j + 1 >= m || st->iters >= st->maxit) {
            st->done = 1;
            st->converged = res <= st->tol;
        } else {
            st->j = j + 1;
        }
    }
    __syncwarp();
    for (int l = lane; l <= j + 1; l += 32) a.H[(int64_t)l * m + j] = shr[l];
}

// ------------------------------------------------------------------ Gram-Schmidt
// Classical Gram-Schmidt with selective reorthogonalisation (DGKS: a second
// pass when ||w_1|| < ||w|| / sqrt(2), gs_second_pass) for Arnoldi column j, in
// three launches with no block ever waiting for another:
//   k_gs_dots    v_j is scaled to unit norm (it was stored as it came; rnorm = 1 /
//                ||v_j|| is k_gm_givens's of the step before) and so is w = far +
//                near part of the product; each block adds its partial dots V_l^H
//                w into column j of H and its partial ||w||^2 into acc (FP64
//                atomics);
//   k_gs_update  w_1 = w - V h and its partial ||w_1||^2; the DGKS test on
//                the sums (||w_1||^2 = ||w||^2 - |h|^2 by Pythagoras; exact
//                enough to decide, since the sums are), and where it asks for a
//                second pass the block adds the dots V_l^H w_1;
//   k_gs_finish  the decision read from the state (k_gs_update's block 0
//                leaves it there); without a second pass w_1 is v_{j+1}; with one
//                h_2 is added to column j of H and w_2 = w_1 - V h_2, with its
//                partial ||w_2||^2, is.  Every block stores its rows of v_{j+1},
//                unnormalised, and the next product's inputs (gs_store).
// Every norm is summed from the vector itself, never estimated (when w_1 is
// mostly rounding noise inside span(V), ||w_1||^2 - |h_2|^2 would cancel to
// nothing and fake a breakdown of the Arnoldi process).
// Every block of k_gs_update takes the same decision from the same FP64
// sums.  Block b owns rows [b R, b R + R) of every vector (R 64 or 128: the basis
// comes from HBM, since each product streams the stored near field through L2, so
// many blocks keep many loads in flight), with FP32 sums within a block.  The
// FP64 sums of the blocks' FP32 partials are exact whenever the partials span
// fewer than 29 binary orders of magnitude, so they do not depend on the
// order in which the blocks add them.  acc ([4]: ||w||^2, ||w_1||^2, ||w_2||^2,
// unused) and h2 alternate between two copies by the parity of j: step j clears
// the copy of step j + 1 (k_gm_start clears both at the start of a cycle, where H
// is cleared too).  The Givens step (k_gm_givens) follows on a side stream.
__device__ __forceinline__ int gs_rows(const GsArgs &a, int64_t &r0)
{
    r0 = (int64_t)blockIdx.x * a.rows;
    const int64_t rem = a.g.n - r0;
    return rem <= 0 ? 0 : (int)(rem < a.rows ? rem : (int64_t)a.rows);
}

__device__ __forceinline__ void atomic_add_c(double2 *p, float2 v)
{
    atomicAdd(&p->x, (double)v.x);
    atomicAdd(&p->y, (double)v.y);
}

// (The basis is read through L1 here and in gs_update: a block reads only
// its own rows, which k_gs_update reads twice, for the update and then the
// second pass's dots.)
// Partial dots sum_{i in block} conj(V_l[i]) ws[i], l <= j, added into
// dst[l * stride]: warp w takes the columns l = w (mod 8), four at a time,
// its lanes the rows, so that every warp keeps several independent loads in
// flight.
__device__ void gs_dots_part(const GsArgs &a, const float2 *ws, int R, int64_t r0, int j, double2 *dst, int64_t stride)
{
    const GmresArgs &g = a.g;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int nwarp = kGsThreads / 32;
    constexpr int kC = 8;     // columns per warp at a time (their loads in flight together)
    for (int l0 = warp; l0 <= j; l0 += kC * nwarp) {
        float2 acc[kC];
#pragma unroll
        for (int u = 0; u < kC; ++u) acc[u] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int i = lane; i < R; i += 32) {
            const float2 y = ws[i];
#pragma unroll
            for (int u = 0; u < kC; ++u) {
                const int l = l0 + u * nwarp;
                if (l <= j) {
                    const float2 x = __ldca(g.V + (int64_t)l * g.n + r0 + i);
                    acc[u].x = fmaf(x.x, y.x, fmaf(x.y, y.y, acc[u].x));
                    acc[u].y = fmaf(x.x, y.y, fmaf(-x.y, y.x, acc[u].y));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kC; ++u) {
            const int l = l0 + u * nwarp;
            const float2 d = warp_sum(acc[u]);
            if (lane == u && l <= j) atomic_add_c(dst + (int64_t)l * stride, d);
        }
    }
}

// The block's sum_{i in block} |ws[i]|^2 added into *nrm.
__device__ void gs_norm_part(const float2 *ws, int R, double *nrm)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int nwarp = kGsThreads / 32;
    __shared__ float red[nwarp];
    float v2 = 0.f;
    for (int i = threadIdx.x; i < R; i += kGsThreads) v2 = fmaf(ws[i].x, ws[i].x, fmaf(ws[i].y, ws[i].y, v2));
    for (int o = 16; o > 0; o >>= 1) v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    if (lane == 0) red[warp] = v2;
    __syncthreads();
    if (warp == 0) {
        float v = lane < nwarp ? red[lane] : 0.f;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(nrm, (double)v);
    }
}

// w_1 = ws - V h (h as FP32 in hs), written back into ws: thread (row rr,
// column group cg) sums the columns l = cg (mod kCg) of its row.
__device__ void gs_update(const GsArgs &a, float2 *ws, const float2 *hs, int R, int64_t r0, int j)
{
    const GmresArgs &g = a.g;
    constexpr int kRowsPerPass = 64, kCg = kGsThreads / kRowsPerPass;
    __shared__ float2 cpart[2][kGsThreads];
    const int cg = threadIdx.x / kRowsPerPass, rr = threadIdx.x % kRowsPerPass;
    // two passes of rows at a time, so each thread has the loads of two rows
    // in flight
    for (int i0 = 0; i0 < R; i0 += 2 * kRowsPerPass) {
        const int ia = i0 + rr, ib = i0 + kRowsPerPass + rr;
        const bool va = ia < R, vb = ib < R;
        float2 acca = make_float2(0.f, 0.f), accb = acca;
        const float2 *pa = g.V + r0 + ia, *pb = g.V + r0 + ib;
#pragma unroll 8
        for (int l = cg; l <= j; l += kCg) {
            const float2 h = hs[l];
            const int64_t o = (int64_t)l * g.n;
            const float2 v = va ? __ldca(pa + o) : make_float2(0.f, 0.f);
            const float2 w = vb ? __ldca(pb + o) : make_float2(0.f, 0.f);
            acca.x = fmaf(h.x, v.x, fmaf(-h.y, v.y, acca.x));
            acca.y = fmaf(h.x, v.y, fmaf(h.y, v.x, acca.y));
            accb.x = fmaf(h.x, w.x, fmaf(-h.y, w.y, accb.x));
            accb.y = fmaf(h.x, w.y, fmaf(h.y, w.x, accb.y));
        }
        cpart[0][threadIdx.x] = acca;
        cpart[1][threadIdx.x] = accb;
        __syncthreads();
        if (cg < 2) {
            const int i = cg == 0 ? ia : ib;
            if (i < R) {
                float2 c = cpart[cg][rr];
#pragma unroll
                for (int q = 1; q < kCg; ++q) {
                    c.x += cpart[cg][rr + q * kRowsPerPass].x;
                    c.y += cpart[cg][rr + q * kRowsPerPass].y;
                }
                ws[i] = make_float2(ws[i].x - c.x, ws[i].y - c.y);
            }
        }
        __syncthreads();
    }
}

// h_l (l <= j) of a column sum as FP32 into hs, and sum_l |h_l|^2 (FP64, the
// same order in every block) returned to every thread.
__device__ double gs_load_h(const double2 *src, int64_t stride, float2 *hs, int j)
{
    __shared__ double s_hh;
    for (int l = threadIdx.x; l <= j; l += kGsThreads) {
        const double2 h = __ldcg(src + (int64_t)l * stride);
        hs[l] = make_float2((float)h.x, (float)h.y);
    }
    if (threadIdx.x < 32) {
        double hh = 0.0;
        for (int l = threadIdx.x; l <= j; l += 32) {
            const double2 h = __ldcg(src + (int64_t)l * stride);
            hh += h.x * h.x + h.y * h.y;
        }
        for (int o = 16; o > 0; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
        if (threadIdx.x == 0) s_hh = hh;
    }
    __syncthreads();
    return s_hh;
}

// DGKS test from the FP64 sums with the classical threshold 1/sqrt(2):
// ||w_1||^2 = ||w||^2 - |h|^2 < ||w||^2 / 2.  (A threshold of 0.1 let the
// FP32 basis lose orthogonality roughly as eps / relres over a GMRES cycle:
// 0.02 after 19 steps, 1 after 53.)
__device__ __forceinline__ bool gs_second_pass(double ww, double hh) { return ww - hh < 0.5 * ww; }

__device__ __forceinline__ void gs_dots_body(const GsArgs &a)
{
    const GmresArgs &g = a.g;
    GmresState *st = g.st;
    int64_t r0;
    const int R = gs_rows(a, r0);
    // w = A v_j (far part g.w + near part) and the state (j, done) are
    // loaded together: one memory round trip before any decision
    constexpr int kWr = kGsMaxRows / kGsThreads;
    float2 wv[kWr];
#pragma unroll
    for (int u = 0; u < kWr; ++u) {
        const int i = threadIdx.x + u * kGsThreads;
        wv[u] = i < R ? cadd(g.w[r0 + i], a.wnear[r0 + i]) : make_float2(0.f, 0.f);
    }
    const int2 jd = __ldcv(reinterpret_cast<const int2 *>(&st->j));   // (j, done)
    const int j = jd.x, done = jd.y;
    if (blockIdx.x == 0 && threadIdx.x == 0) st->skip_prod = done;
    if (done) return;
    // v_j was stored unnormalised (1 / ||v_j|| = st->rnorm, set by k_gm_givens of
    // step j - 1, or 1 by k_gm_start): scale the block's rows of v_j and of
    // the product
    const float sc = __ldcv(&st->rnorm);
    float2 *vj = g.V + (int64_t)j * g.n + r0;
    __shared__ float2 ws[kGsMaxRows];
#pragma unroll
    for (int u = 0; u < kWr; ++u) {
        const int i = threadIdx.x + u * kGsThreads;
        if (i < R) {
            const float2 wsc = cscale(wv[u], sc);
            ws[i] = wsc;
            g.w[r0 + i] = wsc;
            if (j > 0) vj[i] = cscale(vj[i], sc);
        }
    }
    __syncthreads();
    gs_dots_part(a, ws, R, r0, j, g.H + j, g.m);
    gs_norm_part(ws, R, a.acc + 4 * (j & 1));
}

__device__ __forceinline__ void gs_update_body(const GsArgs &a)
{
    const GmresArgs &g = a.g;
    GmresState *st = g.st;
    const int2 jd = __ldcv(reinterpret_cast<const int2 *>(&st->j));
    const int j = jd.x;
    if (jd.y) return;
    int64_t r0;
    const int R = gs_rows(a, r0);
    __shared__ float2 ws[kGsMaxRows];
    __shared__ float2 hs[kMaxRestart + 1];
    for (int i = threadIdx.x; i < R; i += kGsThreads) ws[i] = g.w[r0 + i];
    const double hh = gs_load_h(g.H + j, g.m, hs, j);
    const double ww = __ldcg(a.acc + 4 * (j & 1));
    gs_update(a, ws, hs, R, r0, j);
    for (int i = threadIdx.x; i < R; i += kGsThreads) g.w[r0 + i] = ws[i];
    gs_norm_part(ws, R, a.acc + 4 * (j & 1) + 1);
    const bool need = gs_second_pass(ww, hh);
    // the decision for k_gs_finish (whose block 0 changes column j of H)
    if (blockIdx.x == 0 && threadIdx.x == 0) st->reorth = need;
    if (need) gs_dots_part(a, ws, R, r0, j, a.h2 + (int64_t)(j & 1) * (g.m + 1), 1);
}

// v_{j+1} = ws (unnormalised; its squared norm is in the sums) over the
// block's rows, with the next product's inputs; block 0 keeps the books of
// step j: H column j takes the second pass's h_2 (when there was one), and
// the other parity's sums are cleared for step j + 1.
__device__ void gs_store(const GsArgs &a, const float2 *ws, int R, int64_t r0, int j, bool need)
{
    const GmresArgs &g = a.g;
    GmresState *st = g.st;
    float2 *vn = g.V + (int64_t)(j + 1) * g.n;
    for (int i = threadIdx.x; i < R; i += kGsThreads) {
        const float2 xv = ws[i];
        vn[r0 + i] = xv;
        prep_store(a.next, r0 + i, xv);
    }
    if (blockIdx.x == 0) {
        const double2 *h2 = a.h2 + (int64_t)(j & 1) * (g.m + 1);
        if (need)
            for (int l = threadIdx.x; l <= j; l += kGsThreads) {
                double2 *hp = g.H + (int64_t)l * g.m + j;
                const double2 h = h2[l], h0 = *hp;
                *hp = make_double2(h0.x + h.x, h0.y + h.y);
            }
        double2 *h2n = a.h2 + (int64_t)((j + 1) & 1) * (g.m + 1);
        for (int l = threadIdx.x; l <= j + 1 && l <= g.m; l += kGsThreads) h2n[l] = make_double2(0.0, 0.0);
        if (threadIdx.x < 4) a.acc[4 * ((j + 1) & 1) + threadIdx.x] = 0.0;
        if (threadIdx.x == 0) st->n_reorth += need;
    }
}

__device__ __forceinline__ void gs_finish_body(const GsArgs &a)
{
    const GmresArgs &g = a.g;
    GmresState *st = g.st;
    const int2 jd = __ldcv(reinterpret_cast<const int2 *>(&st->j));
    const int j = jd.x;
    if (jd.y) return;
    int64_t r0;
    const int R = gs_rows(a, r0);
    __shared__ float2 ws[kGsMaxRows];
    __shared__ float2 hs[kMaxRestart + 1];
    for (int i = threadIdx.x; i < R; i += kGsThreads) ws[i] = g.w[r0 + i];
    const bool need = __ldcv(&st->reorth) != 0;      // k_gs_update's decision
    if (need) {
        // second pass: w_2 = w_1 - V h_2 and its partial ||w_2||^2 (summed, as
        // every norm here: when w_1 is mostly rounding noise inside span(V),
        // ||w_1||^2 - |h_2|^2 would cancel to nothing)
        gs_load_h(a.h2 + (int64_t)(j & 1) * (g.m + 1), 1, hs, j);
        gs_update(a, ws, hs, R, r0, j);
        gs_norm_part(ws, R, a.acc + 4 * (j & 1) + 2);
    } else {
        __syncthreads();
    }
    gs_store(a, ws, R, r0, j, need);
}

__global__ void __launch_bounds__(kGsThreads) k_gs_dots(GsArgs a) { gs_dots_body(a); }
__global__ void __launch_bounds__(kGsThreads) k_gs_update(GsArgs a) { gs_update_body(a); }
__global__ void __launch_bounds__(kGsThreads) k_gs_finish(GsArgs a) { gs_finish_body(a); }
__global__ void __launch_bounds__(kGsThreads) k_gs_dots_m(GsPlanes A) { gs_dots_body(A.p[blockIdx.y]); }
__global__ void __launch_bounds__(kGsThreads) k_gs_update_m(GsPlanes A) { gs_update_body(A.p[blockIdx.y]); }
__global__ void __launch_bounds__(kGsThreads) k_gs_finish_m(GsPlanes A)
{
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        // the product kernels skip once every system is done (their flags
        // were set by k_gs_dots_m)
        int all = 1;
        for (int r = 0; r < A.nr; ++r) all &= __ldcv(&A.p[r].g.st->skip_prod) != 0;
        A.p[0].g.st->skip_all = all;
    }
    gs_finish_body(A.p[blockIdx.y]);
}

// Givens step of the column the Gram-Schmidt kernels just formed (one warp
// per plane).
__global__ void k_gm_givens(GsPlanes A)
{
    const GmresArgs &a = A.p[blockIdx.x].g;
    GmresState *st = a.st;
    if (*(volatile int *)&st->done) return;
    // ||v_{j+1}||^2 from the Gram-Schmidt sums (after the second pass when
    // there was one); k_gs_dots of step j + 1 scales v_{j+1} by it
    const int j = st->j;
    const double nn = __ldcg(a.gs_acc + 4 * (j & 1) + (*(volatile int *)&st->reorth ? 2 : 1));
    if (threadIdx.x == 0) st->rnorm = (float)(1.0 / sqrt(nn));
    gm_givens_warp(a, nn, j);
}

// The condition of the WHILE node that runs one Arnoldi cycle on the device
// (each body a few Arnoldi steps, then this kernel, after every step of the
// body, the Givens steps included, has finished): set to 1 while some plane
// is not done and fewer than max_bodies bodies have run, so the loop ends
// even if no plane ever reports done.
__global__ void k_gm_continue(cudaGraphConditionalHandle h, GmresState *st, int nr, int max_bodies)
{
    if (threadIdx.x != 0) return;
    int all = 1;
    for (int r = 0; r < nr; ++r) all &= __ldcv(&st[r].done) != 0;
    const int b = st[0].bodies + 1;
    st[0].bodies = b;
    cudaGraphSetConditional(h, (!all && b < max_bodies) ? 1u : 0u);
}

// Back substitution y = R^{-1} g over ncols columns (FP64), one block per
// plane: column-oriented, each step scales one entry by the reciprocal of its
// diagonal and the lanes of warp 0 update the rest.  The reciprocals 1 / R_ll
// are formed first, all in parallel, so the sequential chain of steps holds no
// division (FP64 division is a long dependent sequence on this part).  The
// triangle is staged packed in shared memory when it fits (smem_cols columns;
// 141 columns from global memory took 212 us, staged 142 us).
__global__ void k_gm_backsolve(GsPlanes A, double2 *__restrict__ yv, int smem_cols)
{
    extern __shared__ double2 tri[];       // row r of the upper triangle from r nc - r (r - 1) / 2
    __shared__ double2 sv[kMaxRestart + 1];
    __shared__ double2 rinv[kMaxRestart + 1];
    const GmresArgs &a = A.p[blockIdx.x].g;
    const double2 *__restrict__ H = a.H, *__restrict__ g = a.g;
    const int m = a.m, nc = a.st->ncols;
    double2 *__restrict__ y = yv + (int64_t)blockIdx.x * (m + 1);
    const int lane = threadIdx.x & 31;
    const bool in_smem = nc <= smem_cols;
    // staging by the whole block (its loads independent of one another),
    // then warp 0 alone runs the sequential steps
    for (int l = threadIdx.x; l < nc; l += blockDim.x) {
        sv[l] = g[l];
        const double2 d = H[(int64_t)l * m + l];
        const double inv = 1.0 / (d.x * d.x + d.y * d.y);
        rinv[l] = make_double2(d.x * inv, -d.y * inv);   // conj(d) / |d|^2
    }
    if (in_smem)
        for (int r = threadIdx.x / 32; r < nc; r += blockDim.x / 32) {
            double2 *row = tri + (r * nc - r * (r - 1) / 2) - r;
            for (int c = r + lane; c < nc; c += 32) row[c] = H[(int64_t)r * m + c];
        }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    for (int l = nc - 1; l >= 0; --l) {
        const double2 ri = rinv[l];
        const double2 sl = sv[l];
        const double2 yl = make_double2(sl.x * ri.x - sl.y * ri.y, sl.x * ri.y + sl.y * ri.x);
        if (lane == 0) y[l] = yl;
        for (int r = lane; r < l; r += 32) {
            const double2 h = in_smem ? tri[r * nc - r * (r - 1) / 2 - r + l] : H[(int64_t)r * m + l];
            sv[r].x -= h.x * yl.x - h.y * yl.y;
            sv[r].y -= h.x * yl.y + h.y * yl.x;
        }
        __syncwarp();
    }
}

// x <- x + sum_l y_l V_l (plane blockIdx.y)
__global__ void k_gm_xupdate(GsPlanes A, float2 *__restrict__ x, const double2 *__restrict__ yv)
{
    __shared__ float2 ys[kMaxRestart + 1];
    const GmresArgs &a = A.p[blockIdx.y].g;
    const float2 *__restrict__ V = a.V;
    const int64_t n = a.n;
    const double2 *__restrict__ y = yv + (int64_t)blockIdx.y * (a.m + 1);
    x += (int64_t)blockIdx.y * n;
    const int nc = a.st->ncols;
    for (int l = threadIdx.x; l < nc; l += blockDim.x) ys[l] = make_float2((float)y[l].x, (float)y[l].y);
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float2 acc = x[i];
    for (int l = 0; l < nc; ++l) acc = cfma(ys[l], V[(int64_t)l * n + i], acc);
    x[i] = acc;
}

// r = b - A x is formed by the caller; here: V_0 = r / ||r|| with ||r|| from
// normpart, and the cycle state is reset (plane blockIdx.y).
__global__ void k_gm_start(GsPlanes A, const float2 *__restrict__ r, int nblk, int first)
{
    const GsArgs &a = A.p[blockIdx.y];
    GmresState *st = a.g.st;
    const int64_t n = a.g.n;
    const int m = a.g.m;
    float2 *__restrict__ V = a.g.V;
    double2 *__restrict__ g = a.g.g;
    r += (int64_t)blockIdx.y * n;
    if (blockIdx.x == 0) {
        // the Gram-Schmidt sums of both parities (see k_gs_dots)
        for (int l = threadIdx.x; l < 2 * (m + 1); l += blockDim.x) a.h2[l] = make_double2(0.0, 0.0);
        if (threadIdx.x < 8) a.acc[threadIdx.x] = 0.0;
        for (int l = threadIdx.x; l <= m; l += blockDim.x) g[l] = make_double2(0.0, 0.0);
    }
    __shared__ double beta_s;
    if (threadIdx.x == 0) {
        double nn = 0.0;
        for (int b = 0; b < nblk; ++b) nn += a.g.normpart[b];
        beta_s = sqrt(nn);
    }
    __syncthreads();
    const double beta = beta_s;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) V[i] = beta > 0.0 ? cscale(r[i], (float)(1.0 / beta)) : make_float2(0.f, 0.f);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (first) st->bnorm = beta;
        st->beta = beta;
        st->j = 0;
        st->rnorm = 1.f;   // v_0 is stored normalised
        st->ncols = 0;
        st->done = 0;
        st->skip_prod = 0;
        // the last cycle may have ended inside a graph body, whose further
        // steps set it: the product of the new v_0 must not skip
        st->skip_all = 0;
        st->converged = 0;
        st->bodies = 0;
        st->resid = st->bnorm > 0.0 ? beta / st->bnorm : 0.0;
        g[0] = make_double2(beta, 0.0);
        if (st->resid <= st->tol) { st->done = 1; st->converged = 1; }
    }
}

// partial ||r||^2 per block (plane blockIdx.y)
__global__ void k_norm_part(GsPlanes A, const float2 *__restrict__ r)
{
    const GmresArgs &a = A.p[blockIdx.y].g;
    const int64_t n = a.n;
    r += (int64_t)blockIdx.y * n;
    double v = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        v += (double)r[i].x * r[i].x + (double)r[i].y * r[i].y;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __shared__ double red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) a.normpart[blockIdx.x] = s;
    }
}

}  // namespace bem
