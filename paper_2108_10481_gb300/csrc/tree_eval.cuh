// Treecode evaluation body (shared by the treecode's own launch and the
// request server's persistent launch). Not part of the C ABI.
#pragma once

#include "internal.h"

namespace pb {

constexpr int TREE_LEAF = 128;     // targets per leaf
constexpr int TREE_REC = 12;       // floats per tree source / proxy record in global memory
constexpr int TREE_DUP = 24;       // floats per record as summed from shared memory: every value twice,
                                   // so that one load gives both halves of a packed f32x2 operand
constexpr int TREE_EVAL_TILE = 128;  // sources staged per round

// kind: the loops of the evaluation. V/K rows: 3 one row without a Yukawa and the other
// without a Laplace term (the direct forms), 0 otherwise; V/K + D/T rows: 1 no Yukawa term,
// 2 V, K, D and T all with a Laplace coefficient, 0 otherwise.
struct TreeCoef {
    float k[2][4];
    float rho[3];  // kind 2: Yukawa over Laplace coefficient of K, D, T
    float kappa;
    float mk2;  // -kappa log2(e)
    int kind;
    int lrow;   // kind 3: the row without a Yukawa term
};

__device__ __forceinline__ float t_rsqrt(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float t_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float2 t_sub2(float2 a, float2 b) {
    float2 d;
    asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n sub.rn.f32x2 rd, ra, rb;\n"
        " mov.b64 {%0, %1}, rd;\n}\n" : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 t_add2(float2 a, float2 b) {
    float2 d;
    asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n add.rn.f32x2 rd, ra, rb;\n"
        " mov.b64 {%0, %1}, rd;\n}\n" : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 t_mul2(float2 a, float2 b) {
    float2 d;
    asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n mul.rn.f32x2 rd, ra, rb;\n"
        " mov.b64 {%0, %1}, rd;\n}\n" : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 t_fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n .reg .b64 ra, rb, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n mov.b64 rc, {%6, %7};\n"
        " fma.rn.f32x2 rd, ra, rb, rc;\n mov.b64 {%0, %1}, rd;\n}\n"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 t_splat(float v) { return make_float2(v, v); }


// One evaluation job: a mesh's tree with its source and proxy records in
// tree order, the kernel coefficients and the partial-sum slices.
struct TreeJob {
    int64_t np;
    int n, nprox;               // proxies per axis and cluster: n^3
    int nsplit;                 // slices of partial sums (the leaves' lists are cut into nsplit shares)
    const int32_t* perm;        // tree index -> point index
    const int32_t* leaf_rng;    // 2 per leaf
    const int32_t* leaf_order;  // leaves by decreasing interaction count
    const int32_t* far_ptr;     // per leaf: its proxied clusters
    const int32_t* far_idx;
    const int32_t* near_ptr;    // per leaf: its directly summed source ranges
    const int32_t* near_rng;
    const float* rec;           // source records in tree order
    const float* prox;          // proxy records per slot
    float* part;                // nsplit x NACC x np
    TreeCoef cf;
};

// Asynchronous 16-byte copies global -> shared (cp.async), committed in groups:
// the staging of the next tile runs while the current one is summed.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The tiles of one leaf's share of its lists, in order: every proxied cluster's
// proxies (far, in tiles of TREE_EVAL_TILE records), then every directly summed
// source range (near, likewise).
struct TreeTiles {
    int32_t f, fe, q, qe;  // list cursors
    int32_t off;           // records done in the current cluster or range
    __device__ __forceinline__ bool next(const TreeJob& T, const float** src, int* cnt, bool* far) {
        constexpr int TILE = TREE_EVAL_TILE;
        if (f < fe) {
            *src = T.prox + ((int64_t)T.far_idx[f] * T.nprox + off) * TREE_REC;
            *cnt = min(TILE / T.n * T.n, T.nprox - off);  // whole columns
            *far = true;
            off += *cnt;
            if (off >= T.nprox) { ++f; off = 0; }
            return true;
        }
        while (q < qe) {
            const int32_t sb = T.near_rng[2 * q], se = T.near_rng[2 * q + 1];
            if (sb + off >= se) { ++q; off = 0; continue; }
            *src = T.rec + (int64_t)(sb + off) * TREE_REC;
            *cnt = min(TILE, se - sb - off);
            *far = false;
            off += TILE;
            if (sb + off >= se) { ++q; off = 0; }
            return true;
        }
        return false;
    }
};

// The proxies of a cluster are a tensor grid: a column of N has one x and one y, so that two of
// the three differences and their squares are taken once for it, and its T sums' x and y parts by
// one multiply-add of the column's sum. `cols` columns of staged records, those from g0 on in
// steps of NQ, onto the sums acc of two targets X. A staged record, every value twice: z, the
// charges (V/K rows: a, b of kind 3's two kernels or of both rows; V/K + D/T rows: S, a, b of the
// phi row, C, N), and at 20 x, y.
struct TreeConst {
    float2 kap, mk2, rhoD, rhoT, c10, c11, c12, c13;
};
template <int MODE, int KIND, int NQ, int N, int NS>
__device__ __forceinline__ void far_columns(const float* cur, int cols, int g0, const float2& X0, const float2& X1,
                                            const float2& X2, const TreeConst& k, float2 (&acc)[NS]) {
    constexpr bool YUK = KIND != 1;
    for (int c = g0; c < cols; c += NQ) {
        const float* col = cur + TREE_DUP * N * c;
        const float4 xy = *reinterpret_cast<const float4*>(col + 20);
        const float2 d0 = t_sub2(X0, make_float2(xy.x, xy.y)), d1 = t_sub2(X1, make_float2(xy.z, xy.w));
        const float2 rho2 = t_fma2(d0, d0, t_mul2(d1, d1));
        float2 st = t_splat(0.f);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float4* z4 = reinterpret_cast<const float4*>(col + TREE_DUP * i);
            const float4 a = z4[0], b = z4[1];
            const float2 d2 = t_sub2(X2, make_float2(a.x, a.y));
            const float2 r2 = t_fma2(d2, d2, rho2);
            const float2 rinv = make_float2(t_rsqrt(r2.x), t_rsqrt(r2.y));
            float2 e = t_splat(0.f), g = e;
            if (YUK) {
                const float2 arg = t_mul2(t_mul2(r2, rinv), k.mk2);
                e = make_float2(t_ex2(arg.x), t_ex2(arg.y));
            }
            if (MODE == 0) {
                if (KIND == 3) {
                    acc[0] = t_fma2(rinv, make_float2(a.z, a.w), acc[0]);
                    acc[1] = t_fma2(t_mul2(e, rinv), make_float2(b.x, b.y), acc[1]);
                } else {
                    const float4 dd = z4[2];
                    acc[0] = t_fma2(rinv, t_fma2(e, make_float2(b.x, b.y), make_float2(a.z, a.w)), acc[0]);
                    acc[1] = t_fma2(rinv, t_fma2(e, make_float2(dd.x, dd.y), make_float2(b.z, b.w)), acc[1]);
                }
            } else {
                const float4 cc = z4[2], dd = z4[3], ee = z4[4];
                const float2 ri2 = t_mul2(rinv, rinv);
                float2 kt = rinv, kd = rinv;
                acc[0] = t_fma2(rinv, make_float2(b.x, b.y), acc[0]);
                if (YUK) {
                    g = t_mul2(e, rinv);
                    acc[0] = t_fma2(g, make_float2(b.z, b.w), acc[0]);
                    const float2 gw = t_fma2(k.kap, e, g);
                    if (KIND == 2) {
                        kt = t_fma2(k.rhoT, gw, rinv);
                        kd = t_fma2(k.rhoD, g, rinv);
                    } else {
                        kt = t_fma2(k.c13, gw, t_mul2(k.c12, rinv));
                        kd = t_fma2(k.c11, g, t_mul2(k.c10, rinv));
                    }
                }
                const float2 ts = t_mul2(kt, t_mul2(ri2, make_float2(a.z, a.w)));
                st = i == 0 ? ts : t_add2(st, ts);
                acc[3] = t_fma2(ts, d2, acc[3]);
                acc[4] = t_fma2(kd, make_float2(cc.x, cc.y), acc[4]);
                acc[5] = t_fma2(kd, make_float2(cc.z, cc.w), acc[5]);
                acc[6] = t_fma2(kd, make_float2(dd.x, dd.y), acc[6]);
                if (YUK) {
                    acc[7] = t_fma2(g, make_float2(dd.z, dd.w), acc[7]);
                    acc[8] = t_fma2(g, make_float2(ee.x, ee.y), acc[8]);
                    acc[9] = t_fma2(g, make_float2(ee.z, ee.w), acc[9]);
                }
            }
        }
        if (MODE == 1) {
            acc[1] = t_fma2(st, d0, acc[1]);
            acc[2] = t_fma2(st, d1, acc[2]);
        }
    }
}

// One leaf of targets and one split of its lists, on 64 NQ threads: a thread
// holds two targets (the leaf's i-th and (i + 64)-th points) in packed f32x2
// arithmetic; the NQ thread groups of 64 take every NQ-th source of each staged
// tile and add their sums through shared memory at the end, group 0 adding
// groups 1 .. NQ-1 in that order. Far: proxies of the well-separated clusters
// (kernel G with the interpolated charges). Near: the other sources directly,
// with the direct pair kernel's arithmetic (identical points skipped). Tiles
// are staged in two buffers by asynchronous copies, the next one in flight
// while the current one is summed; before it is summed a tile is copied once
// more inside shared memory with every value twice (TREE_DUP floats per
// record), which keeps the records in global memory (and L2) at 48 bytes, and
// with the charges that only meet constant kernel coefficients combined with
// them there (per record a, b with a + e b the Laplace + Yukawa weight, e =
// exp(-kappa r)), which takes 3 to 6 operations off every interaction.
// `tile` holds at least TREE_EVAL_TILE x (2 TREE_REC + TREE_DUP) floats and
// (NQ - 1) x NACC x TREE_LEAF floats. Every thread of the group calls it (it
// synchronises the CTA) and returns with no copy in flight.
//
// FP32 operations per interaction (the packed pipe is the limit, with the loads of the splatted
// records close behind), proxy and direct: V/K rows 7 (kind 3) or 8, and 19; V/K + D/T rows 21 and 32
// (kind 2), 11 and 20 (kind 1), 23 and 36 (kind 0), with 4 or 6 more a column of proxies (every
// proxy by itself: 11, 12; 26, 16, 29). Sums kept per target (NS): V/K rows the two rows' proxy
// sums (kind 3: the Laplace and the Yukawa one), then the four sums of the direct pairs; V/K +
// D/T rows phi, T, C, B, scaled at the end by kind. Columns: 116,160 points, direct form: 948 -> 813 us;
// 661,500 points, Juffer form: 11.9 -> 10.5 ms.
template <int MODE, int KIND, int NQ>
__device__ __forceinline__ void tree_leaf_body(const TreeJob& T, int leaf, int sp, float* tile) {
    constexpr int NACC = MODE == 0 ? 2 : 10;
    constexpr int NS = MODE == 0 ? 6 : 10;
    constexpr bool YUK = KIND != 1;
    constexpr int TILE = TREE_EVAL_TILE;
    constexpr int HALF = TREE_LEAF / 2;
    constexpr int NTH = HALF * NQ;
    const int nsp = T.nsplit;
    const int32_t fb0 = T.far_ptr[leaf], nfar = T.far_ptr[leaf + 1] - fb0;
    const int32_t qb0 = T.near_ptr[leaf], nnear = T.near_ptr[leaf + 1] - qb0;
    const int32_t fb = fb0 + (int32_t)((int64_t)nfar * sp / nsp), fe = fb0 + (int32_t)((int64_t)nfar * (sp + 1) / nsp);
    const int32_t qb = qb0 + (int32_t)((int64_t)nnear * sp / nsp), qe = qb0 + (int32_t)((int64_t)nnear * (sp + 1) / nsp);
    const int64_t np = T.np;
    float* part = T.part + (int64_t)sp * NACC * np;
    const float* rec = T.rec;
    const int32_t tb = T.leaf_rng[2 * leaf], te = T.leaf_rng[2 * leaf + 1];
    const int grp = (int)threadIdx.x / HALF;
    const int32_t ti0 = tb + (int32_t)(threadIdx.x % HALF), ti1 = ti0 + HALF;
    const bool live0 = ti0 < te, live1 = ti1 < te;
    float2 X0 = t_splat(0.f), X1 = X0, X2 = X0;
    if (live0) {
        X0.x = rec[TREE_REC * (int64_t)ti0];
        X1.x = rec[TREE_REC * (int64_t)ti0 + 1];
        X2.x = rec[TREE_REC * (int64_t)ti0 + 2];
    }
    if (live1) {
        X0.y = rec[TREE_REC * (int64_t)ti1];
        X1.y = rec[TREE_REC * (int64_t)ti1 + 1];
        X2.y = rec[TREE_REC * (int64_t)ti1 + 2];
    }
    const TreeCoef& cf = T.cf;
    const float2 c02 = t_splat(cf.k[0][2]), c03 = t_splat(cf.k[0][3]), c10 = t_splat(cf.k[1][0]),
                 c11 = t_splat(cf.k[1][1]), c12 = t_splat(cf.k[1][2]), c13 = t_splat(cf.k[1][3]),
                 kap = t_splat(cf.kappa), mk2 = t_splat(cf.mk2), rhoK = t_splat(cf.rho[0]),
                 rhoD = t_splat(cf.rho[1]), rhoT = t_splat(cf.rho[2]);
    // charges of a staged record: the phi row's coefficients (kind 3: of the row each kernel belongs to)
    const int rl = KIND == 3 ? cf.lrow : 0, ry = KIND == 3 ? 1 - cf.lrow : 0;
    const float pscale = KIND == 1 || KIND == 2 ? cf.k[0][2] : 1.0f;  // K's Laplace coefficient, carried by p (and N)
    float2 acc[NS];
    for (int k = 0; k < NS; ++k) acc[k] = t_splat(0.f);
    const TreeConst kc = {kap, mk2, rhoD, rhoT, c10, c11, c12, c13};
    int turn = 0;
    const bool any = live0;  // the first target of a thread is live whenever the second is
    TreeTiles it = {fb, fe, qb, qe, 0};
    const float* src = nullptr;
    int cnt = 0, cnt_next = 0;
    bool far = false, far_next = false;
    bool have = it.next(T, &src, &cnt, &far);
    __syncthreads();  // the buffers may still be read by the caller's previous work
    if (have) {
        for (int k = threadIdx.x; k < cnt * TREE_REC / 4; k += NTH) cp_async16(tile + 4 * k, src + 4 * k);
    }
    cp_async_commit();
    for (int buf = 0; have; buf ^= 1) {
        const float* nsrc = nullptr;
        const bool have_next = it.next(T, &nsrc, &cnt_next, &far_next);
        if (have_next) {
            float* nb = tile + (buf ^ 1) * TILE * TREE_REC;
            for (int k = threadIdx.x; k < cnt_next * TREE_REC / 4; k += NTH) cp_async16(nb + 4 * k, nsrc + 4 * k);
        }
        cp_async_commit();
        cp_async_wait<1>();  // this thread's copies of the current tile have landed
        __syncthreads();     // and every thread's; the duplicated tile's last readers are done
        float* dup = tile + 2 * TILE * TREE_REC;
        for (int r = threadIdx.x; r < cnt; r += NTH) {
            // a record as summed: the charges that only ever meet the kernel coefficients
            // combined with them once here (Laplace and Yukawa parts a + e b, e = exp(-kappa r))
            const float4* rp = reinterpret_cast<const float4*>(tile + buf * TILE * TREE_REC + TREE_REC * r);
            const float4 u0 = rp[0], u1 = rp[1], u2 = rp[2];
            float v[TREE_REC] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w, u2.x, u2.y, u2.z, u2.w};
            const float s_ = v[3];
            if (far) {  // as far_columns reads them
                const float q_ = v[4], x_ = v[0], y_ = v[1];
                v[0] = v[2];
                if (MODE == 0) {
                    v[1] = fmaf(cf.k[rl][2], q_, cf.k[rl][0] * s_);
                    v[2] = fmaf(cf.k[ry][3], q_, cf.k[ry][1] * s_);
                    v[3] = fmaf(cf.k[1][2], q_, cf.k[1][0] * s_);
                    v[4] = fmaf(cf.k[1][3], q_, cf.k[1][1] * s_);
                } else {
                    v[1] = s_;
                    v[2] = fmaf(cf.k[0][2], q_, cf.k[0][0] * s_);
                    v[3] = fmaf(cf.k[0][3], q_, cf.k[0][1] * s_);
#pragma unroll
                    for (int k = 4; k < 10; ++k) v[k] = k < 7 ? v[k + 1] : pscale * v[k + 1];
                }
                v[10] = x_;
                v[11] = y_;
            } else if (MODE == 1) {  // x, s, p, c, (a, b) of the phi row's single layer
#pragma unroll
                for (int k = 4; k < 7; ++k) v[k] *= pscale;
                v[10] = cf.k[0][0] * s_;
                v[11] = cf.k[0][1] * s_;
            }
            float4* d4 = reinterpret_cast<float4*>(dup + TREE_DUP * r);
#pragma unroll
            for (int h = 0; h < TREE_REC / 2; ++h) d4[h] = make_float4(v[2 * h], v[2 * h], v[2 * h + 1], v[2 * h + 1]);
        }
        __syncthreads();
        const float* cur = dup;
        if (far) {
            const int cols = cnt / T.n, g0 = (grp + turn) % NQ;
            turn = (turn + NQ - cols % NQ) % NQ;  // the groups' shares even out over the tiles
            if (any) {
                switch (T.n) {
                    case 3: far_columns<MODE, KIND, NQ, 3>(cur, cols, g0, X0, X1, X2, kc, acc); break;
                    case 4: far_columns<MODE, KIND, NQ, 4>(cur, cols, g0, X0, X1, X2, kc, acc); break;
                    case 5: far_columns<MODE, KIND, NQ, 5>(cur, cols, g0, X0, X1, X2, kc, acc); break;
                    case 6: far_columns<MODE, KIND, NQ, 6>(cur, cols, g0, X0, X1, X2, kc, acc); break;
                    case 7: far_columns<MODE, KIND, NQ, 7>(cur, cols, g0, X0, X1, X2, kc, acc); break;
                    default: far_columns<MODE, KIND, NQ, 8>(cur, cols, g0, X0, X1, X2, kc, acc); break;
                }
            }
        } else if (any) {
#pragma unroll 2
            for (int j = grp; j < cnt; j += NQ) {
                const float4* y4 = reinterpret_cast<const float4*>(cur + TREE_DUP * j);
                const float4 a = y4[0], b = y4[1], c = y4[2], dd = y4[3];
                const float2 y3 = make_float2(b.z, b.w), p0 = make_float2(c.x, c.y), p1 = make_float2(c.z, c.w),
                             p2 = make_float2(dd.x, dd.y);
                const float2 d0 = t_sub2(X0, make_float2(a.x, a.y)), d1 = t_sub2(X1, make_float2(a.z, a.w)),
                             d2 = t_sub2(X2, make_float2(b.x, b.y));
                const float2 r2 = t_fma2(d0, d0, t_fma2(d1, d1, t_mul2(d2, d2)));
                const float2 rinv = make_float2(r2.x > 0.f ? t_rsqrt(r2.x) : 0.f, r2.y > 0.f ? t_rsqrt(r2.y) : 0.f);
                float2 g = t_splat(0.f), gw = g;
                if (YUK) {
                    const float2 arg = t_mul2(t_mul2(r2, rinv), mk2);
                    const float2 e = make_float2(t_ex2(arg.x), t_ex2(arg.y));
                    g = t_mul2(e, rinv);
                    gw = t_fma2(kap, e, g);
                }
                const float2 ri2 = t_mul2(rinv, rinv);
                const float2 dp = t_mul2(ri2, t_fma2(d0, p0, t_fma2(d1, p1, t_mul2(d2, p2))));
                if (MODE == 0) {
                    acc[2] = t_fma2(rinv, y3, acc[2]);
                    acc[3] = t_fma2(rinv, dp, acc[3]);
                    acc[4] = t_fma2(g, y3, acc[4]);
                    acc[5] = t_fma2(gw, dp, acc[5]);
                } else {
                    const float4 ee = y4[4], ff = y4[5];
                    float2 kk = rinv, kt = rinv, kd = rinv;
                    acc[0] = t_fma2(rinv, make_float2(ff.x, ff.y), acc[0]);
                    if (YUK) {
                        acc[0] = t_fma2(g, make_float2(ff.z, ff.w), acc[0]);
                        if (KIND == 2) {
                            kk = t_fma2(rhoK, gw, rinv);
                            kt = t_fma2(rhoT, gw, rinv);
                            kd = t_fma2(rhoD, g, rinv);
                        } else {
                            kk = t_fma2(c03, gw, t_mul2(c02, rinv));
                            kt = t_fma2(c13, gw, t_mul2(c12, rinv));
                            kd = t_fma2(c11, g, t_mul2(c10, rinv));
                        }
                    }
                    acc[0] = t_fma2(kk, dp, acc[0]);
                    const float2 ts = t_mul2(kt, t_mul2(ri2, y3));
                    acc[1] = t_fma2(ts, d0, acc[1]);
                    acc[2] = t_fma2(ts, d1, acc[2]);
                    acc[3] = t_fma2(ts, d2, acc[3]);
                    acc[4] = t_fma2(kd, make_float2(dd.z, dd.w), acc[4]);
                    acc[5] = t_fma2(kd, make_float2(ee.x, ee.y), acc[5]);
                    acc[6] = t_fma2(kd, make_float2(ee.z, ee.w), acc[6]);
                    if (YUK) {
                        acc[7] = t_fma2(g, p0, acc[7]);
                        acc[8] = t_fma2(g, p1, acc[8]);
                        acc[9] = t_fma2(g, p2, acc[9]);
                    }
                }
            }
        }
        have = have_next;
        cnt = cnt_next;
        far = far_next;
    }
    cp_async_wait<0>();  // nothing in flight (the last group is empty)
    // the sums -> the rows' accumulators
    float2 out[NACC];
    if (MODE == 0) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float2 f = KIND == 3 ? (r == cf.lrow ? acc[0] : acc[1]) : acc[r];
            out[r] = t_fma2(t_splat(cf.k[r][0]), acc[2],
                            t_fma2(t_splat(cf.k[r][2]), acc[3],
                                   t_fma2(t_splat(cf.k[r][1]), acc[4], t_fma2(t_splat(cf.k[r][3]), acc[5], f))));
        }
    } else {
        out[0] = acc[0];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            out[1 + k] = KIND == 0 ? acc[1 + k] : t_mul2(c12, acc[1 + k]);
            out[4 + k] = KIND == 0 ? acc[4 + k] : t_mul2(c10, acc[4 + k]);
            out[7 + k] = KIND == 2 ? t_mul2(t_splat(1.0f / cf.k[0][2]), acc[7 + k]) : acc[7 + k];
        }
    }
    // the other groups' sums join group 0's, in group order
    __syncthreads();
    const int tl = (int)threadIdx.x % HALF;
    if (grp > 0) {
        float* slot = tile + (grp - 1) * NACC * TREE_LEAF;
        for (int k = 0; k < NACC; ++k) {
            slot[k * TREE_LEAF + tl] = out[k].x;
            slot[k * TREE_LEAF + HALF + tl] = out[k].y;
        }
    }
    __syncthreads();
    if (grp == 0) {
        for (int g2 = 1; g2 < NQ; ++g2) {
            const float* slot = tile + (g2 - 1) * NACC * TREE_LEAF;
            for (int k = 0; k < NACC; ++k) {
                out[k].x += slot[k * TREE_LEAF + tl];
                out[k].y += slot[k * TREE_LEAF + HALF + tl];
            }
        }
        if (live0) {
            const int64_t pt = T.perm[ti0];
            for (int k = 0; k < NACC; ++k) part[(int64_t)k * np + pt] = out[k].x;
        }
        if (live1) {
            const int64_t pt = T.perm[ti1];
            for (int k = 0; k < NACC; ++k) part[(int64_t)k * np + pt] = out[k].y;
        }
    }
    __syncthreads();  // the buffer is free for the caller
}

// host side (tree.cu): the mesh's tree built if needed, its source records and
// proxy charges computed on stream s for the far-field plan fp and the
// coefficients x, and the evaluation job described (partial sums in the mesh's
// ws_part, nsplit slices).
int tree_prepare(const pb_mesh* m, const FarPlan& fp, const double* x, bool need_u, bool need_v, TreeJob* job,
                 cudaStream_t s);
// pairs of one application (direct + proxy) and leaves, for cost estimates
int64_t tree_interactions(const pb_mesh* m);
int64_t tree_leaves(const pb_mesh* m);

}  // namespace pb
