// lbm_resident.cuh -- many time steps of small domains in one launch.
//
// A domain that fits on the chip is cut into tiles, one per CTA of one
// cooperative launch, and every CTA keeps its tile's f* in shared memory for
// all the steps of the launch; only the edges of the tiles cross between SMs,
// through L2. The node arithmetic is that of lbm_step.cuh operation for
// operation, so the populations are bit for bit those of the step kernel.
//
// What bounds small domains in the step kernel is not bandwidth but the chain
// of each step: a launch, the staging of the first rows, the row pipeline. Here
// a step is two CTA barriers, and the launch, the staging and the trip of the
// whole state through L2 fall away. Measured (us per step, before -> now):
// 128x64 FP32 6.7 -> 0.9, 1024x128 FP32 deviations 8.2 -> 2.8 (8.2 -> 2.3 in
// FP32), 1024x256 FP16 deviations 8.5 -> 4.1, 1024x512 FP32 11.0 -> 5.3.
//
// A round is K steps and one exchange. The tile holds a halo of 2 K nodes (a
// step reaches two nodes: one for the pull, one for psi); step m of the round
// recomputes what of the halo the later ones need:
//   1. pull rows and columns 2 m + 1 .. from each side: rho, rho u, and psi
//      into shared memory; barrier;
//   2. forces and collision of all but the outermost of these, f* written back
//      in place (every pull of the step has been made); barrier;
//   3. after the last step of a round the tile's nodes within 2 K of its edge
//      are published and the halo is received.
// K = 1 costs the least arithmetic; small tiles take 2 or 4 and pay the trip
// through L2 (about 0.9 us) once for several steps (128x64: 1.4 us a step at
// K = 1, 1.0 at 2, 0.95 at 4). The plan (res_plan) picks the tiling and K.
//
// One warp works on one row of up to 32 columns, so every shared-memory access
// is to consecutive elements; a flat split of the tile's nodes over the
// threads had 44% bank conflicts and ran at 82% of the shared-memory rate. Rows
// go to the warps in turn, which spreads the slower rows along a wall
// (1024x512: 6.8 -> 5.9 us against blocks of rows). Two rows in straight line
// per warp (spills) and pairs of columns per thread (half the warps) were
// slower: 4.2 -> 5.0 and 4.2 -> 5.0 us at 1024x256. Counters of 64 steps in one
// launch (128x64, 1024x128 and 1024x512): issue slots 38, 51 and 63% busy, the
// shared-memory pipe 14, 34 and 39%, bank conflicts 3, 9 and 15% of its
// wavefronts; the rest is waiting, at barriers first in the smallest domain.
//
// Exchange: a published node is NB records of 16 bytes, three (or fewer)
// values and the round's tag, each stored and loaded as one 128-bit access, so
// a record whose tag matches is complete: no fence, no separate flag, one
// trip through L2. Records of one kind lie together, so that a warp reads
// consecutive ones (a node's records side by side: 5.9 -> 9.0 us at 1024x512).
// Tags count steps over the lifetime of the exchange buffer and are not reused;
// two buffers alternate. A tile overwrites a record two rounds after it
// published it, when it has received the next round from every neighbour,
// which had then read the record: every tile publishes all its edge nodes,
// solid ones too, and receives them all, so two tiles that share a halo always
// wait for each other. Waits are bounded as in the step kernel: on timeout a
// thread raises the error flag and waits no more.
#pragma once

#include "lbm_step.cuh"

namespace lbm {

// 16-byte records per published node: 9 FP32 values, or rho* and 8 16-bit
// deviations
__host__ __device__ constexpr int res_records(int st) { return is16(st) ? 2 : 3; }

// Shared memory of a resident tile: per row of kResP nodes (the tile's and
// its halo's columns) the planes of the storage form, psi and, in the
// deviation forms, the sum of a node's own deviations; then the table of the
// tile's halo nodes. One warp works on one row (the 32 columns but the two
// outermost), so every shared-memory access is to 32 consecutive elements.
constexpr int kResP = 34;
// Threads per CTA at most with J rows per warp; two such CTAs fit on an SM (56
// registers a thread for J <= 2, 64 above).
__host__ __device__ constexpr int res_max_threads(int j) { return j == 1 ? 576 : j == 2 ? 544 : 512; }
constexpr int kResMaxRows = 5;  // rows per warp at most (tau = 1; 2 otherwise)
// floats per row; plane 0 (and all nine of plain storage) comes first
template <int ST> __host__ __device__ constexpr int res_row_floats()
{
    return ST == kF32 ? 10 * kResP : ST == kF32Dev ? 11 * kResP : 3 * kResP + 8 * kResP / 2;
}
template <int ST> __host__ __device__ constexpr int res_psi() { return ST == kF32 ? 9 * kResP : kResP; }
constexpr int kResDown = 2 * kResP, kResDev = 3 * kResP;  // deviation forms: own sum, first deviation plane
// rows and halo nodes of the largest tile
template <int ST> __host__ __device__ constexpr size_t res_smem_bytes(int rows, int nhalo)
{
    return size_t(rows) * res_row_floats<ST>() * sizeof(float) + size_t(nhalo) * 2 * sizeof(int);
}

// Nodes within dep of the edge of a w x h tile, and the index of such a node
// in the tile's published records: the first dep rows, the last dep rows,
// then the 2 dep outer columns of the rows between (all nodes row by row when
// nothing is left inside).
__host__ __device__ inline int res_edge_nodes(int w, int h, int dep)
{
    return (w <= 2 * dep || h <= 2 * dep) ? w * h : 2 * dep * (w + h - 2 * dep);
}
__host__ __device__ inline int res_edge_index(int x, int y, int w, int h, int dep)
{
    if (w <= 2 * dep || h <= 2 * dep || y < dep) return y * w + x;
    if (y >= h - dep) return (y - (h - dep) + dep) * w + x;
    return 2 * dep * w + (y - dep) * 2 * dep + (x < dep ? x : x - (w - 2 * dep));
}
// tile i of n along a side of len nodes covers [res_cut(i), res_cut(i + 1))
__host__ __device__ inline int res_cut(int i, int n, int len) { return int((long long)i * len / n); }
__host__ __device__ inline int res_owner(int x, int n, int len)
{
    int i = int((long long)x * n / len);
    while (res_cut(i + 1, n, len) <= x) ++i;
    while (res_cut(i, n, len) > x) --i;
    return i;
}

__device__ __forceinline__ void put_record(uint4* p, uint32_t a, uint32_t b, uint32_t c, uint32_t tag)
{
    asm volatile(
        "{\n\t.reg .b64 lo, hi;\n\t.reg .b128 v;\n\tmov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\t"
        "mov.b128 v, {lo, hi};\n\tst.relaxed.gpu.global.b128 [%0], v;\n\t}" ::"l"(p),
        "r"(a), "r"(b), "r"(c), "r"(tag)
        : "memory");
}
__device__ __forceinline__ uint4 get_record(const uint4* p)
{
    uint4 r;
    asm volatile(
        "{\n\t.reg .b64 lo, hi;\n\t.reg .b128 v;\n\tld.relaxed.gpu.global.b128 v, [%4];\n\tmov.b128 {lo, hi}, v;\n\t"
        "mov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
        : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
        : "l"(p)
        : "memory");
    return r;
}

// Sum of a node's own deviations (d1, d2), (d3, d4), (d5, d6), (d7, d8) in
// pull_dev's order.
__device__ __forceinline__ float dev_own_sum(const float2 (&q)[4])
{
    const float2 a = add2(q[0], q[1]), b = add2(q[2], q[3]);
    return (a.x + a.y) + (b.x + b.y);
}

// Pull node x of the resident rows m, c, p (y - 1, y, y + 1): pull_smem or
// pull_dev operation for operation (the sum of the node's own deviations was
// stored with them). WALLS = false leaves the bounce-back out: right unless
// rho comes out NaN, which a solid node or source always makes it.
template <int ST, bool WALLS, typename N>
__device__ __forceinline__ void res_pull(const float* __restrict__ m, const float* __restrict__ c,
                                         const float* __restrict__ p, int x, bool need_g, N& n)
{
    using T = typename StoreT<ST>::T;
    constexpr int P = kResP;
    constexpr int opp[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
    const float r0 = c[x];
    n.sb = 0;
    if constexpr (WALLS) {
        n.solid = is_solid(r0);
        if (n.solid) {
            n.rho = n.jx = n.jy = 0.f;
            return;
        }
    } else {
        n.solid = false;
    }
    if constexpr (ST == kF32) {
        float v[9];
        v[0] = r0;
        v[1] = c[1 * P + x - 1];
        v[2] = m[2 * P + x];
        v[3] = c[3 * P + x + 1];
        v[4] = p[4 * P + x];
        v[5] = m[5 * P + x - 1];
        v[6] = m[6 * P + x + 1];
        v[7] = p[7 * P + x + 1];
        v[8] = p[8 * P + x - 1];
        if constexpr (WALLS) {
            float own[9];
#pragma unroll
            for (int a = 1; a < 9; ++a) own[a] = c[a * P + x];
#pragma unroll
            for (int a = 1; a < 9; ++a) {
                const bool w = is_solid(v[a]);
                n.sb |= w ? 1u << a : 0u;
                v[a] = w ? own[opp[a]] : v[a];
            }
        }
        n.rho = ((v[0] + (v[1] + v[3])) + (v[2] + v[4])) + ((v[5] + v[7]) + (v[6] + v[8]));
#pragma unroll
        for (int a = 0; a < 9; ++a) n.f[a] = v[a];
        n.jx = (v[1] - v[3]) + (v[5] - v[7]) + (v[8] - v[6]);
        n.jy = (v[2] - v[4]) + (v[5] - v[7]) + (v[6] - v[8]);
    } else {
        constexpr float U = RawScale<T>::unscale, S = RawScale<T>::scale;
        auto dv = [](const float* row, int col, int a) {
            return to_raw(reinterpret_cast<const T*>(row + kResDev)[(a - 1) * P + col]);
        };
        float2 rA = make_float2(c[x - 1], m[x - 1]), rB = make_float2(c[x + 1], p[x + 1]);
        float2 rC = make_float2(m[x], m[x + 1]), rD = make_float2(p[x], p[x - 1]);
        float2 dA = make_float2(dv(c, x - 1, 1), dv(m, x - 1, 5)), dB = make_float2(dv(c, x + 1, 3), dv(p, x + 1, 7));
        float2 dC = make_float2(dv(m, x, 2), dv(m, x + 1, 6)), dD = make_float2(dv(p, x, 4), dv(p, x - 1, 8));
        if constexpr (WALLS) {
            float rs[9] = {0.f, rA.x, rC.x, rB.x, rD.x, rA.y, rC.y, rB.y, rD.y};
            float d[9] = {0.f, dA.x, dC.x, dB.x, dD.x, dA.y, dC.y, dB.y, dD.y};
            float own[9];
#pragma unroll
            for (int a = 1; a < 9; ++a) own[a] = dv(c, x, a);
#pragma unroll
            for (int a = 1; a < 9; ++a) {
                const bool w = is_solid(rs[a]);
                n.sb |= w ? 1u << a : 0u;
                rs[a] = w ? r0 : rs[a];
                d[a] = w ? own[opp[a]] : d[a];
            }
            rA = make_float2(rs[1], rs[5]); rB = make_float2(rs[3], rs[7]);
            rC = make_float2(rs[2], rs[6]); rD = make_float2(rs[4], rs[8]);
            dA = make_float2(d[1], d[5]); dB = make_float2(d[3], d[7]);
            dC = make_float2(d[2], d[6]); dD = make_float2(d[4], d[8]);
        }
        const float down = c[kResDown + x];
        const float2 r0s = splat(r0);
        const float2 qa = sub2(rA, r0s), qb = sub2(rB, r0s), qc = sub2(rC, r0s), qd = sub2(rD, r0s);
        const float2 q = add2(add2(qa, qb), add2(qc, qd));
        constexpr float w1 = 1.f / 9.f, w2 = 1.f / 36.f;
        const float2 ds = add2(add2(dA, dB), add2(dC, dD));
        const float dsrc = ds.x + ds.y;
        const float drho = fmaf(w1, q.x, fmaf(w2, q.y, (dsrc - down) * U));
        n.rho = r0 + drho;
        const float2 er = sub2(rA, rB), fr = sub2(rC, rD), ed = sub2(dA, dB), fd = sub2(dC, dD);
        float2 jd = make_float2((ed.x + ed.y) - fd.y, (fd.x + ed.y) + fd.y);
        if constexpr (U != 1.f) jd = mul2(jd, splat(U));
        const float2 j = fma2(splat(w1), make_float2(er.x, fr.x),
                              fma2(splat(w2), make_float2(er.y - fr.y, er.y + fr.y), jd));
        n.jx = j.x;
        n.jy = j.y;
        if (need_g) {
            const float2 wS = make_float2(w1 * S, w2 * S), dr = splat(drho);
            const float2 gA = fma2(wS, sub2(qa, dr), dA), gB = fma2(wS, sub2(qb, dr), dB);
            const float2 gC = fma2(wS, sub2(qc, dr), dC), gD = fma2(wS, sub2(qd, dr), dD);
            n.g[1] = gA.x; n.g[5] = gA.y; n.g[3] = gB.x; n.g[7] = gB.y;
            n.g[2] = gC.x; n.g[6] = gC.y; n.g[4] = gD.x; n.g[8] = gD.y;
        }
        n.g[0] = 0.f;
    }
}

constexpr uint32_t kResWaitLimit = 1u << 20;  // polls of a record before giving up (about a second)

// Poll a published node's records (stride apart) until all carry the tag; false
// after the last poll (the first, for a thread that has given up before). The
// caller raises the error flag and gives up: with that in here and `alive` by
// reference, the step loop's code was 1.4% slower (101 steps of 301x67).
template <int NB>
__device__ __forceinline__ bool poll_records(const uint4* q, int stride, uint32_t tag, bool alive, uint4 (&r)[NB])
{
    bool ok = false;
    for (uint32_t i = 0; i < kResWaitLimit; ++i) {
        ok = true;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            r[b] = get_record(q + b * stride);
            ok = ok && r[b].w == tag;
        }
        if (ok || !alive) break;
    }
    return ok;
}

// A node's stored state as 32-bit words: 9 populations, rho* and 8
// deviations, or rho* and 4 pairs of 16-bit deviations.
template <int ST> constexpr int kResWords = is16(ST) ? 5 : 9;

template <int ST> __device__ __forceinline__ void res_put_node(float* row, int x, const uint32_t (&v)[kResWords<ST>])
{
    if constexpr (ST == kF32) {
#pragma unroll
        for (int a = 0; a < 9; ++a) row[a * kResP + x] = __uint_as_float(v[a]);
    } else {
        using T = typename StoreT<ST>::T;
        row[x] = __uint_as_float(v[0]);
        float2 q[4];
        if constexpr (is16(ST)) {
            uint16_t* d = reinterpret_cast<uint16_t*>(row + kResDev);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                d[(2 * k) * kResP + x] = uint16_t(v[1 + k]);
                d[(2 * k + 1) * kResP + x] = uint16_t(v[1 + k] >> 16);
                q[k] = unpack_raw2<T>(v[1 + k]);
            }
        } else {
#pragma unroll
            for (int a = 1; a < 9; ++a) row[kResDev + (a - 1) * kResP + x] = __uint_as_float(v[a]);
#pragma unroll
            for (int k = 0; k < 4; ++k) q[k] = make_float2(__uint_as_float(v[1 + 2 * k]), __uint_as_float(v[2 + 2 * k]));
        }
        row[kResDown + x] = dev_own_sum(q);
    }
}

template <int ST> __device__ __forceinline__ void res_get_node(const float* row, int x, uint32_t (&v)[kResWords<ST>])
{
    v[0] = __float_as_uint(row[x]);
    if constexpr (is16(ST)) {
        const uint16_t* d = reinterpret_cast<const uint16_t*>(row + kResDev);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            v[1 + k] = uint32_t(d[(2 * k) * kResP + x]) | uint32_t(d[(2 * k + 1) * kResP + x]) << 16;
    } else {
#pragma unroll
        for (int a = 1; a < 9; ++a) v[a] = __float_as_uint(row[(a + (ST == kF32 ? 0 : 2)) * kResP + x]);
    }
}

template <int ST> __device__ __forceinline__ void put_node_records(uint4* q, int stride, const uint32_t (&v)[kResWords<ST>], uint32_t tag)
{
    put_record(q, v[0], v[1], v[2], tag);
    if constexpr (is16(ST)) {
        put_record(q + stride, v[3], v[4], 0u, tag);
    } else {
        put_record(q + stride, v[3], v[4], v[5], tag);
        put_record(q + 2 * stride, v[6], v[7], v[8], tag);
    }
}

// nsteps steps of one tile, a halo of 2 K nodes exchanged every K steps (the
// last round may be shorter). J: rows per warp at most. exch: 2 x (CTAs of
// the launch) x records x edge_cap records. out may be in where the launch has
// an exchange (nsteps > K): a tile writes its final state after it has received
// records from every tile that reads it, which those publish after their loads.
template <int ST, bool T1, int J>
__device__ __forceinline__ void run_resident(const Geom& g, const Phys& p, const float* in,
                                             float* out, int tx, int ty, int first, int tile, int K,
                                             uint4* exch, int parity_stride, int edge_cap, uint32_t tag0, int nsteps,
                                             int* err, unsigned char* smem)
{
    using T = typename StoreT<ST>::T;
    using PT = std::conditional_t<ST == kF32, Pulled, PulledDev>;
    constexpr int NB = res_records(ST), NW = kResWords<ST>, RS = res_row_floats<ST>(), PSI = res_psi<ST>();
    const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, warp = t >> 5, nw = nt >> 5;
    const int ti = tile % tx, tj = tile / tx, dep = 2 * K, dsh = K == 4 ? 4 : K + 1;  // 2 dep = 1 << dsh (K = 1, 2, 4)
    const int x0 = res_cut(ti, tx, g.nx), w = res_cut(ti + 1, tx, g.nx) - x0;
    const int y0 = res_cut(tj, ty, g.ny), h = res_cut(tj + 1, ty, g.ny) - y0;
    const int W = w + 2 * dep, H = h + 2 * dep;  // the tile and its halo (W <= kResP)
    float* s = reinterpret_cast<float*>(smem);
    int2* halo = reinterpret_cast<int2*>(s + H * RS);  // (record, place in s)
    auto wrap = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };

    for (int k = t; k < H * RS; k += nt) s[k] = 0.f;
    __syncthreads();
    // the state of the tile and its halo
    for (int r = warp; r < H; r += nw) {
        const int gy = wrap(y0 - dep + r, g.ny);
        for (int x = lane; x < W; x += 32) {
            const size_t o = size_t(gy) * g.pitch + wrap(x0 - dep + x, g.nx);
            uint32_t v[NW];
            v[0] = __float_as_uint(in[o]);
            if constexpr (is16(ST)) {
                const uint4 q = reinterpret_cast<const uint4*>(in + g.plane)[o];
                v[1] = q.x; v[2] = q.y; v[3] = q.z; v[4] = q.w;
            } else {
#pragma unroll
                for (int a = 1; a < 9; ++a) v[a] = __float_as_uint(in[size_t(a) * g.plane + o]);
            }
            res_put_node<ST>(s + r * RS, x, v);
        }
    }
    __syncthreads();
    // where each halo node comes from, and where it goes unless it is solid
    const int nhalo = W * H - w * h;
    for (int k = t; k < nhalo; k += nt) {
        int ex, ey;
        if (k < 2 * dep * W) {
            ey = k / W;
            ex = k % W;
            if (ey >= dep) ey += h;
        } else {
            const int r = k - 2 * dep * W;
            ey = dep + r / (2 * dep);
            ex = r % (2 * dep);
            if (ex >= dep) ex += w;
        }
        const int gx = wrap(x0 - dep + ex, g.nx), gy = wrap(y0 - dep + ey, g.ny);
        const int oi = res_owner(gx, tx, g.nx), oj = res_owner(gy, ty, g.ny);
        const int ox = res_cut(oi, tx, g.nx), oy = res_cut(oj, ty, g.ny);
        const int e = res_edge_index(gx - ox, gy - oy, res_cut(oi + 1, tx, g.nx) - ox, res_cut(oj + 1, ty, g.ny) - oy, dep);
        const bool s_solid = is_solid(s[ey * RS + ex]);
        halo[k] = make_int2((first + oj * tx + oi) * NB * edge_cap + e, s_solid ? -1 : (ey * RS) << 6 | ex);
    }
    const int mine = (first + tile) * NB * edge_cap;
    const int x = 1 + lane;  // this thread's column in every row
    // every node is within dep of the tile's edge
    const bool all = w <= 2 * dep || h <= 2 * dep;
    bool alive = true, odd = false;
    __syncthreads();

#pragma unroll 1
    for (int done = 0; done < nsteps;) {
        const int steps = min(K, nsteps - done);
        const bool last_round = done + steps == nsteps;
        const uint32_t tag = tag0 + uint32_t(done);
        uint4* const ex = exch + (odd ? parity_stride : 0);
        uint4* const out_rec = ex + mine;
        odd = !odd;
#pragma unroll 1
        for (int m = K - steps; m < K; ++m) {
            // rows lo .. hi - 1 and columns lo .. W - lo - 1 are pulled, all
            // but the outermost of them collided; rows go to the warps in
            // turn, so that the slower rows along a wall are spread
            const int lo = 1 + 2 * m, hi = H - lo, r0 = lo + warp;
            float* row0 = s + r0 * RS;
            PT n[J];
#pragma unroll
            for (int j = 0; j < J; ++j) {
                if (r0 + j * nw >= hi) break;
                float* c = row0 + j * nw * RS;
                res_pull<ST, false>(c - RS, c, c + RS, x, !T1 && p.tau != 1.f, n[j]);
                if (isnan(n[j].rho)) res_pull<ST, true>(c - RS, c, c + RS, x, !T1 && p.tau != 1.f, n[j]);
                c[PSI + x] = pseudopotential(p, n[j]);
            }
            __syncthreads();
            const bool cols = x > lo && x < W - lo - 1;
            const bool publish = m == K - 1 && !last_round;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int r = r0 + j * nw;
                if (!(r > lo && r < hi - 1)) continue;
                float* c = row0 + j * nw * RS;
                // a solid node's result is not used
                const float2 F = node_force(n[j], c + PSI - RS, c + PSI, c + PSI + RS, x, p);
                const float rinv = rcp_approx(n[j].rho);
                uint32_t v[NW];
                if constexpr (ST == kF32) {
                    float fs[9];
                    relax_node<T1>(n[j], F, rinv, p, fs);
#pragma unroll
                    for (int a = 0; a < 9; ++a) v[a] = __float_as_uint(fs[a]);
                } else {
                    float2 q[4];
                    relax_dev<T, T1>(n[j], F, rinv, p, q);
                    v[0] = __float_as_uint(n[j].rho);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if constexpr (is16(ST)) {
                            v[1 + k] = pack_raw2<T>(q[k]);
                        } else {
                            v[1 + 2 * k] = __float_as_uint(q[k].x);
                            v[2 + 2 * k] = __float_as_uint(q[k].y);
                        }
                    }
                }
                const int ly = r - dep;
                if (publish && (all || ly < dep || ly >= h - dep)) {
                    const int e = (all || ly < dep ? ly : ly - h + 2 * dep) * w + x - dep;
                    if (cols) put_node_records<ST>(out_rec + e, edge_cap, v, tag);
                }
                if (cols && !n[j].solid) res_put_node<ST>(c, x, v);
            }
            if (m < K - 1) {
                __syncthreads();
            } else if (!last_round && !all) {
                // the side columns of this warp's other rows, read back from
                // shared memory so that the rows share the instructions
                __syncwarp();
                const int cc = lane & (2 * dep - 1), lx = cc < dep ? cc : cc + w - 2 * dep;
                for (int ly = r0 - dep + (lane >> dsh) * nw; ly < h - dep; ly += (32 >> dsh) * nw) {
                    if (ly < dep) continue;
                    uint32_t v[NW];
                    res_get_node<ST>(s + (ly + dep) * RS, lx + dep, v);
                    put_node_records<ST>(out_rec + 2 * dep * w + ((ly - dep) << dsh) + cc, edge_cap, v, tag);
                }
            }
        }
        done += steps;
        if (last_round) break;
        for (int k = t; k < nhalo; k += nt) {
            const int2 hk = halo[k];
            const uint4* q = ex + hk.x;
            uint4 r[NB];
            if (!poll_records(q, edge_cap, tag, alive, r) && alive) {
                atomicOr(err, 1);
                alive = false;
            }
            uint32_t v[NW];
            if constexpr (is16(ST)) {
                v[0] = r[0].x; v[1] = r[0].y; v[2] = r[0].z; v[3] = r[NB - 1].x; v[4] = r[NB - 1].y;
            } else {
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    v[3 * b] = r[b].x;
                    v[3 * b + 1] = r[b].y;
                    v[3 * b + 2] = r[b].z;
                }
            }
            if (hk.y >= 0) res_put_node<ST>(s + (hk.y >> 6), hk.y & 63, v);
        }
        __syncthreads();
    }
    // the final state (solid nodes hold their sentinel in both buffers)
    __syncthreads();
    for (int ly = warp; ly < h; ly += nw) {
        if (lane >= w) continue;
        uint32_t v[NW];
        res_get_node<ST>(s + (ly + dep) * RS, lane + dep, v);
        if (v[0] == kSolidBits) continue;
        const size_t og = size_t(y0 + ly) * g.pitch + x0 + lane;
        out[og] = __uint_as_float(v[0]);
        if constexpr (is16(ST)) {
            reinterpret_cast<uint4*>(out + g.plane)[og] = make_uint4(v[1], v[2], v[3], v[4]);
        } else {
#pragma unroll
            for (int a = 1; a < 9; ++a) out[size_t(a) * g.plane + og] = __uint_as_float(v[a]);
        }
    }
}

// One domain, every CTA one tile.
template <int ST, bool T1, int J>
__global__ void __launch_bounds__(res_max_threads(J), 2)
    resident_kernel(const float* in, float* out, Geom g, Phys p, int tx, int ty, int K,
                    uint4* exch, int parity_stride, int edge_cap, uint32_t tag0, int nsteps, int* err)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    run_resident<ST, T1, J>(g, p, in, out, tx, ty, 0, blockIdx.x, K, exch, parity_stride, edge_cap, tag0, nsteps, err,
                            smem_raw);
}

// Several domains: CTA i works on tile ctas[i].y of domain ctas[i].x, whose
// tiling is shape (tx, ty, first CTA); buf[parity] is read and buf[parity_out]
// written.
template <int ST, bool T1, int J>
__global__ void __launch_bounds__(res_max_threads(J), 2)
    resident_batch_kernel(const DomainDev* __restrict__ doms, const int4* __restrict__ shape,
                          const int2* __restrict__ ctas, int parity, int parity_out, int K, uint4* exch, int parity_stride,
                          int edge_cap, uint32_t tag0, int nsteps, int* err)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ Geom g;
    __shared__ Phys p;
    const int2 c = ctas[blockIdx.x];
    const DomainDev& d = doms[c.x];
    if (threadIdx.x == 0) {
        g = d.g;
        p = d.p;
    }
    __syncthreads();
    const int4 sh = shape[c.x];
    run_resident<ST, T1, J>(g, p, d.buf[parity], d.buf[parity_out], sh.x, sh.y, sh.z, c.y, K, exch, parity_stride,
                            edge_cap, tag0, nsteps, err, smem_raw);
}

}  // namespace lbm
