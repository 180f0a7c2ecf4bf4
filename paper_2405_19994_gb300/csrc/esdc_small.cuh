// The whole step of a small mesh as one persistent cooperative launch (FP64 path,
// single handles).
//
// Below about one node per resident thread a step is a chain of K (M + 1) node
// evaluations and K M solves whose kernels each have next to nothing to do: a
// 32x32 sheet spent 650 us per step in 76 dependent launches of 2 to 10 us.
// What bounds such a step is latency, and three kinds of it:
//  * launches: here one thread owns a node's V row for the whole step, and there
//    is one launch;
//  * grid barriers (2700 cycles on 152 SMs) and the L2 trips around them: blocks
//    exchange values through 16-byte cells {value, tag} written and read in one
//    piece.  A reader polls the very cells it needs until their tag is the one of
//    this phase, so a Chebyshev iteration waits for its neighbours only (about
//    1400 cycles instead of 5300 for store, barrier and load);
//  * FP64 issue: one warp gets an FP64 instruction through every 64 cycles,
//    whatever its lanes and dependences, and an SM one every 19 (four warps
//    76).  A node's work is therefore split over `roles` warps (the V row and
//    the auxiliaries; the gates in equal shares), and the gates' warps work
//    while the V warps solve: a gate's row needs V_{i-1} only.
//
// The V row is solved in correction form, x = x_w + e with (I - g A) e = r, where
// x_w is the warm start and r its residual (node_v's R0 form: no stencil on
// x_w, f_I is linear in V).  e is orders below V, so the rounding of the solve
// is too.
//  * DCT-II handles: dense cosine products, split by parity (element i and
//    n-1-i enter as their sum or difference, so an axis of length n costs n/2
//    FMAs and one addition per value and direction): 17 FP64 instructions in a
//    row at n = 32, where the FFT's stages are about 55.
//  * otherwise: the Chebyshev semi-iteration of k_cheb on the same interval with
//    the same stop test; x, r, d in registers, only d is exchanged.
//
// Measured per step, launch sequence -> this kernel: 32x32 HH sheet (M 3, K 4) 650 ->
// 191 us, 101x75 HH sheet 757 -> 365 us, 500-node HH cable (M 6, K 8) 2.46 -> 0.91 ms,
// 48x40x10 SYN19 slab (M 4, K 6) 2.37 -> 1.21 ms.  A Chebyshev iteration is then about
// 3100 cycles (1700 of them waiting for a neighbour's cell), a node's V row 8000.
//
// Every wait is bounded (1 s, or esdc_debug_barrier's limit): a thread whose wait
// runs out raises TIMEOUT and waits for nothing more, so the launch ends.
#pragma once
#include <atomic>

#include "esdc_cg_common.cuh"
#include "esdc_kernels.cuh"

#define ESDC_SMALL_TAB 64
#define ESDC_SMALL_MINIT 3           // iterations that run before the starting residual's sum is asked for
constexpr int kSmallStageDoubles = 18 * 1024;   // matrices of the axes that a block stages in shared memory

typedef unsigned long long SmallTag;
struct __align__(16) SmallCell {
    double v;
    SmallTag tag;
};

struct SmallArgs {
    int K, fuse1, dct, layers, fourth;
    int lgnb, roles;                 // log2 of the nodes per block; warps' roles per node
    int maxit;
    double tol2;
    double rho0[ESDC_MMAX + 1];      // warm-start weights of sweep 0
    double g[ESDC_MMAX + 1];         // dt d_i times the operator's scale
    double *G0, *G1, *yout;
    SmallCell* cells;                // [ESDC_SMALL_BUFS][N] (Chebyshev: the first two)
    SmallCell* part;                 // [2][2][gridDim.x] partial sums
    unsigned* bar;
    int *status, *log;
    int log_len;
    // DCT-II
    SmallAxis ax[3];
    int stage;                       // doubles of the axes' matrices staged in shared memory (0: read from global)
    double* winv;                    // [M][ld]: spectral weight / (1 - g_i mu)
    const double *ex, *ey, *ez;
    double wgt;
    // Chebyshev: 1/theta and per iteration ca, cb, 4 q^{2 (k + 1)}
    double inv_theta[ESDC_MMAX + 1];
    double ca[ESDC_MMAX + 1][ESDC_SMALL_TAB], cb[ESDC_MMAX + 1][ESDC_SMALL_TAB], qq[ESDC_MMAX + 1][ESDC_SMALL_TAB];
};

namespace {

__device__ __forceinline__ void cell_put(SmallCell* c, double v, SmallTag tag)
{
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}"
                 :: "l"(c), "l"(__double_as_longlong(v)), "l"(tag) : "memory");
}

__device__ __forceinline__ void cell_load(const SmallCell* c, double& v, SmallTag& tag)
{
    long long b;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(b), "=l"(tag) : "l"(c) : "memory");
    v = __longlong_as_double(b);
}

struct SmallWait {
    const unsigned* bar;
    int* flags;
    bool dead;
};

// Every 256 polls: whether this wait has lasted too long.
__device__ __noinline__ bool small_expired(const unsigned* bar, unsigned long long& t0)
{
    if (!t0) { t0 = global_ns(); return false; }
    const unsigned us = __ldcg(bar + 3);
    return global_ns() - t0 > (us ? 1000ull * us : kWaitLimitNs);
}

// v[e] = the value of cell at[e] once its tag is `tag`, for the entries of mask.
template <int NB>
__device__ __forceinline__ void cells_get(const SmallCell* c, const int (&at)[NB], unsigned mask, SmallTag tag,
                                          double (&v)[NB], SmallWait& w)
{
    unsigned need = mask, spins = 0;
    unsigned long long t0 = 0;
    while (need) {
        SmallTag t[NB];
        double x[NB];
#pragma unroll
        for (int e = 0; e < NB; ++e)
            if ((need >> e) & 1u) cell_load(c + at[e], x[e], t[e]);
#pragma unroll
        for (int e = 0; e < NB; ++e)
            if (((need >> e) & 1u) && t[e] == tag) {
                v[e] = x[e];
                need &= ~(1u << e);
            }
        if (!need || w.dead) break;
        if ((++spins & 255u) == 0 && small_expired(w.bar, t0)) {
            w.dead = true;
            atomicOr(w.flags, ESDC_FLAG_TIMEOUT);
        }
    }
}

__device__ __forceinline__ double cell_get(const SmallCell* c, int at, SmallTag tag, SmallWait& w)
{
    const int a[1] = {at};
    double v[1] = {0.0};
    cells_get<1>(c, a, 1u, tag, v, w);
    return v[0];
}

// Barrier among the V warps (the first nb threads of the block).
__device__ __forceinline__ void v_sync(int nb)
{
    if (nb == 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"r"(nb) : "memory");
}

// The grid's sums of NV values over the V threads, the same bits in every block:
// warp trees, the warps in order, the blocks in order of a lane's stride, a tree.
// post: stores the block's sums in its cells (tag = the reduction's number);
// take: waits for every block's.  Reduction n + 2 reuses the cells of n: a block
// posts n + 1 after it has taken n, and n + 2 after every block has posted n + 1.
template <int NV>
__device__ __forceinline__ void sums_post(const double (&v)[NV], SmallCell* part, SmallTag n, int tl, int nb)
{
    __shared__ double sh[NV][16];
    SmallCell* cell = part + (size_t)(n & 1) * 2 * gridDim.x + blockIdx.x;
    const int lane = tl & 31, w = tl >> 5, nw = nb >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = v[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) {
            if (nw == 1) cell_put(cell + (size_t)k * gridDim.x, x, n);
            else sh[k][w] = x;
        }
    }
    if (nw == 1) return;
    v_sync(nb);
    if (tl < NV) {
        double x = sh[tl][0];
        for (int k = 1; k < nw; ++k) x += sh[tl][k];
        cell_put(cell + (size_t)tl * gridDim.x, x, n);
    }
}

template <int NV>
__device__ __forceinline__ void sums_take(const SmallCell* part, SmallTag n, int tl, int nb, double (&tot)[NV],
                                          SmallWait& wt)
{
    __shared__ double res[2];
    if (tl < 32) {
        const SmallCell* cell = part + (size_t)(n & 1) * 2 * gridDim.x;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const SmallCell* c = cell + (size_t)k * gridDim.x;
            double x = 0.0;
            for (unsigned b0 = tl; b0 < gridDim.x; b0 += 128) {
                int at[4];
                unsigned mask = 0;
                double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    at[e] = b0 + 32 * e;
                    if (b0 + 32 * e < gridDim.x) mask |= 1u << e;
                }
                cells_get<4>(c, at, mask, n, v, wt);
                x += (v[0] + v[1]) + (v[2] + v[3]);
            }
            __syncwarp();
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if (tl == 0) res[k] = x;
        }
    }
    v_sync(nb);
#pragma unroll
    for (int k = 0; k < NV; ++k) tot[k] = res[k];
    v_sync(nb);
}

// The operator's neighbours of a node: A v = sum_q cf_q (v_q - v_p) with the faces
// (scalar, field and layered), the layered operator's in-plane diagonals (entries
// 6..9) or the fourth-order stencil (12 entries, mirrored).
struct SmallStencil {
    double cf[12], cs;               // cs: the sum of cf
    int q[12];
    unsigned mask;                   // entries with a neighbour other than p
};

__device__ __noinline__ void small_stencil(const MeshDev& m, int p, bool has, NodeIdx n, SmallStencil& o)
{
    o.cs = 0.0;
    o.mask = 0;
    for (int e = 0; e < 12; ++e) { o.cf[e] = 0.0; o.q[e] = p; }
    if (!has) return;
    const int idx[3] = {n.ix, n.iy, n.iz}, len[3] = {m.nx, m.ny, m.nz}, st[3] = {1, m.nx, m.nx * m.ny};
    auto add = [&](int e, int q, double c) {
        o.q[e] = q;
        o.cf[e] = c;
        if (q != p) {
            o.mask |= 1u << e;
            o.cs += c;
        }
    };
    if (m.order == 4) {
        for (int a = 0; a < 3; ++a) {
            if (len[a] == 1) continue;
            for (int e = 0; e < 4; ++e) {
                const int off = e < 2 ? e - 2 : e - 1;                           // -2, -1, 1, 2
                add(4 * a + e, p + (esdc_mirror(idx[a] + off, len[a]) - idx[a]) * st[a],
                    (off == -1 || off == 1 ? 16.0 : -1.0) * (m.ih2 * (1.0 / 12.0)));
            }
        }
        return;
    }
    for (int e = 0; e < 6; ++e) {
        const int a = e >> 1, off = (e & 1) ? 1 : -1, j = idx[a] + off;
        if (j < 0 || j >= len[a]) continue;
        const int q = p + off * st[a];
        double c = m.ih2;
        if (m.sig) c = (0.5 * m.ih2) * (__ldg(m.sig + p) + __ldg(m.sig + q));
        else if (m.lay) c = __ldg(m.lay + (a < 2 ? a * m.nz + n.iz : 3 * m.nz + (off > 0 ? n.iz : n.iz - 1)));
        add(e, q, c);
    }
    if (m.lay) {
        const double cd = __ldg(m.lay + 2 * m.nz + n.iz);
        for (int e = 0; e < 4; ++e) {
            const int ox = (e & 1) ? 1 : -1, oy = (e & 2) ? 1 : -1, jx = n.ix + ox, jy = n.iy + oy;
            if (jx < 0 || jx >= m.nx || jy < 0 || jy >= m.ny) continue;
            add(6 + e, p + ox + oy * m.nx, ox == oy ? cd : -cd);
        }
    }
}

// A V at the node from the neighbours' cells.
__device__ __noinline__ double small_lap(const SmallStencil& st, const SmallCell* c, SmallTag tag, double vp, SmallWait& w)
{
    double v[12], s = 0.0;
#pragma unroll
    for (int e = 0; e < 12; ++e) v[e] = vp;
    cells_get<12>(c, st.q, st.mask, tag, v, w);
#pragma unroll
    for (int e = 0; e < 12; ++e)
        if ((st.mask >> e) & 1u) s = fma(st.cf[e], v[e] - vp, s);
    return s;
}

// ---------------------------------------------------------------- Chebyshev
// The solve's correction to the warm start; tag: the last tag this thread's cells
// carry (the direction of tag t is in buffer t & 1: a thread publishes t + 1 after
// it has read its neighbours' t, which they published after reading its t - 1).
// FIRST: the starting residual's sum is asked for before any iteration (a solve by
// itself may have none to do), not during the first ones.  mute: this block does not
// post that sum (esdc_debug_barrier).
template <int NB, bool FIRST = false, class Args = SmallArgs>
__device__ __noinline__ double small_cheb(const SmallStencil& st, const Args& s, int N, int i, int slot, int p,
                                          bool has, int tl, int nb, const NodeSolve& so, SmallTag& tag, SmallTag& nred,
                                          SmallWait& wt, bool mute = false)
{
    double cf[NB];
    int q[NB];
#pragma unroll
    for (int e = 0; e < NB; ++e) { cf[e] = st.cf[e]; q[e] = st.q[e]; }
    const unsigned mask = st.mask;
    const double g = s.g[i], cs = st.cs;
    double r = has ? so.r : 0.0, d = r * s.inv_theta[i], x = 0.0;
    ++tag;
    if (has) cell_put(s.cells + (tag & 1) * N + p, d, tag);
    {
        const double v[2] = {r * r, has ? so.b * so.b : 0.0};
        ++nred;
        if (!FIRST || !mute) sums_post<2>(v, s.part, nred, tl, nb);
    }
    const int first = FIRST ? 0 : (s.maxit < ESDC_SMALL_MINIT ? s.maxit : ESDC_SMALL_MINIT);
    int it = 0, check_at = first;
    double stop = 0.0, tot0 = 0.0;
    bool done = false, bad = false;
    auto ask = [&]() {
        // the iterations the bound asks for: the first k with 2 q^k ||r_0|| <= tol ||b||
        double tot[2];
        sums_take<2>(s.part, nred, tl, nb, tot, wt);
        tot0 = tot[0];
        stop = s.tol2 * tot[1];
        bad = !isfinite(tot[0]) || !isfinite(stop);
        __shared__ int s_need;
        if (tl < 32) {
            int need = 0;
            if (!(tot[0] <= stop)) {
                need = ESDC_SMALL_TAB;
                for (int k0 = 0; k0 < ESDC_SMALL_TAB; k0 += 32) {
                    const unsigned hit = __ballot_sync(0xffffffffu, s.qq[i][k0 + tl] * tot[0] <= stop);
                    if (hit) { need = k0 + __ffs(hit); break; }
                }
            }
            if constexpr (FIRST) {                        // past the table by the formula
                if (need == ESDC_SMALL_TAB && stop > 0.0) {
                    const double kd = ceil(log(0.5 * sqrt(stop / tot[0])) / s.log_q);
                    need = kd < (double)s.maxit ? (int)kd : s.maxit;
                } else if (need == ESDC_SMALL_TAB) {
                    need = s.maxit;                       // tol 0: to the cap
                }
            }
            if (tl == 0) s_need = need;
        }
        v_sync(nb);
        check_at = s_need > first ? s_need : first;
        if (check_at > s.maxit) check_at = s.maxit;
    };
    if (FIRST) {
        ask();
        done = tot0 <= stop;
    }
    while (!FIRST || !(done || bad)) {
        const int ki = it < ESDC_SMALL_TAB ? it : ESDC_SMALL_TAB - 1;
        if (has) {
            double dv[NB];
#pragma unroll
            for (int e = 0; e < NB; ++e) dv[e] = 0.0;
            cells_get<NB>(s.cells + (tag & 1) * N, q, mask, tag, dv, wt);
            double t = cs * d;
#pragma unroll
            for (int e = 0; e < NB; ++e)
                if ((mask >> e) & 1u) t = fma(-cf[e], dv[e], t);
            r -= fma(g, t, d);
            x += d;
            d = fma(s.ca[i][ki], d, s.cb[i][ki] * r);
        }
        ++it;
        if (!FIRST && it == first) {
            ask();
            if (bad) break;
        }
        if (it == check_at) {
            const double v[1] = {r * r};
            double rr[1];
            sums_post<1>(v, s.part, ++nred, tl, nb);
            sums_take<1>(s.part, nred, tl, nb, rr, wt);
            bad = !isfinite(rr[0]);
            done = rr[0] <= stop;
            if (bad || done || it == s.maxit) break;
            check_at = it + 2 < s.maxit ? it + 2 : s.maxit;     // rounding left it short: two more, then check
        }
        ++tag;
        if (has) cell_put(s.cells + (tag & 1) * N + p, d, tag);
    }
    if (blockIdx.x == 0 && tl == 0) {
        s.status[0] = it;
        if (slot < s.log_len) s.log[slot] = it;
        if (bad) atomicOr(wt.flags, ESDC_FLAG_NONFINITE);
        else if (!done) atomicOr(wt.flags, ESDC_FLAG_CG_MAXIT);
    }
    return x;
}

// ---------------------------------------------------------------- DCT-II
// Exchange buffers of the transforms.  One tag per solve and buffer suffices: a
// cell's next value depends, through the solve's last stage, on the outputs of
// every thread that reads its present one.
enum { kBufR = 0, kBufX, kBufY, kBufZ, kBufW, kBufE, kBufV, ESDC_SMALL_BUFS };

// One axis for lines [L0, L0 + nl) (element stride inner).  MODE 0: forward;
// 1: inverse; 2: forward, times scale, inverse.  in: the cells read, or nullptr
// for values in sr (the block's own x lines).  out: the cells written, or nullptr:
// the value of work item tl (the thread's own node) is returned.  sa, sb: nl * n
// doubles of shared memory each.
template <int MODE>
__device__ __forceinline__ double small_axis(const SmallAxis& A, const double* F, const double* B, double* sa, double* sb,
                                             const double* sr, const SmallCell* in, SmallCell* out, SmallTag tag,
                                             const double* scale, int inner, int L0, int nl, int tl, int nb, SmallWait& wt)
{
    const int n = A.n, hp = A.hp, h = n >> 1, lg = (n & (n - 1)) == 0 ? 31 - __clz(n) : -1;
    double mine = 0.0;
    auto base = [&](int l) {
        const int L = L0 + l;
        if (inner == 1) return L * n;
        const int o = L / inner;
        return o * n * inner + (L - o * inner);
    };
    auto line = [&](int w) { return lg >= 0 ? w >> lg : w / n; };
    if (MODE != 1) {
        for (int w = tl; w < nl * hp; w += nb) {
            const int l = inner == 1 ? w / hp : w % nl, i = inner == 1 ? w - l * hp : w / nl, b = base(l);
            double v[2] = {0.0, 0.0};
            if (in) {
                const int at[2] = {b + i * inner, b + (n - 1 - i) * inner};
                cells_get<2>(in, at, i < h ? 3u : 1u, tag, v, wt);
            } else {
                v[0] = sr[l * n + i];
                v[1] = sr[l * n + n - 1 - i];
            }
            if (i < h) {
                sa[l * n + i] = v[0] + v[1];
                sa[l * n + n - 1 - i] = v[0] - v[1];
            } else {
                sa[l * n + i] = v[0];                    // the middle of an odd axis: even modes only
            }
        }
        v_sync(nb);
        for (int w = tl; w < nl * n; w += nb) {
            const int l = line(w), k = w - l * n;
            const double* v = sa + l * n + ((k & 1) ? n - 1 : 0);
            const int dir = (k & 1) ? -1 : 1, cnt = (k & 1) ? h : hp;
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
            int i = 0;
            for (; i + 4 <= cnt; i += 4) {
                s0 = fma(v[dir * i], F[i * n + k], s0);
                s1 = fma(v[dir * (i + 1)], F[(i + 1) * n + k], s1);
                s2 = fma(v[dir * (i + 2)], F[(i + 2) * n + k], s2);
                s3 = fma(v[dir * (i + 3)], F[(i + 3) * n + k], s3);
            }
            for (; i < cnt; ++i) s0 = fma(v[dir * i], F[i * n + k], s0);
            const double X = (s0 + s1) + (s2 + s3);
            const int at = base(l) + k * inner;
            if (MODE == 0) cell_put(out + at, X, tag);
            else sb[l * n + k] = X * __ldcg(scale + at);
        }
    } else {
        for (int w = tl; w < nl * n; w += nb) {
            const int l = inner == 1 ? line(w) : w % nl, k = inner == 1 ? w - l * n : w / nl;
            sb[l * n + k] = cell_get(in, base(l) + k * inner, tag, wt);
        }
    }
    v_sync(nb);
    if (MODE == 0) return 0.0;
    // even half e_t (t < hp) and odd half o_t (t < h) of the outputs t and n-1-t
    for (int w = tl; w < nl * n; w += nb) {
        const int l = line(w), t = w - l * n;
        const int odd = t >= hp, c = odd ? t - hp : t;
        const double* X = sb + l * n;
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
        int k = odd;
        for (; k + 6 < n; k += 8) {
            s0 = fma(X[k], B[k * hp + c], s0);
            s1 = fma(X[k + 2], B[(k + 2) * hp + c], s1);
            s2 = fma(X[k + 4], B[(k + 4) * hp + c], s2);
            s3 = fma(X[k + 6], B[(k + 6) * hp + c], s3);
        }
        for (; k < n; k += 2) s0 = fma(X[k], B[k * hp + c], s0);
        sa[w] = (s0 + s1) + (s2 + s3);
    }
    v_sync(nb);
    for (int w = tl; w < nl * n; w += nb) {
        const int l = inner == 1 ? line(w) : w % nl, j = inner == 1 ? w - l * n : w / nl;
        const int t = j < hp ? j : n - 1 - j;
        const double e = sa[l * n + t], o = t < h ? sa[l * n + hp + t] : 0.0;
        const double y = j < hp ? e + o : e - o;
        if (out) cell_put(out + base(l) + j * inner, y, tag);
        else mine = y;
    }
    v_sync(nb);
    return mine;
}

template <int MODE>
__device__ __noinline__ double small_axis_all(const SmallArgs& s, const MeshDev& m, int a, double* mats, double* work,
                                              const double* sr, const SmallCell* in, SmallCell* out, SmallTag tag,
                                              const double* scale, int tl, int nb, SmallWait& wt)
{
    const SmallAxis& A = s.ax[a];
    const int n = A.n, inner = a == 0 ? 1 : (a == 1 ? m.nx : m.nx * m.ny), lines = m.N / n;
    const int nl = nb >= n ? nb / n : 1;
    const double *F = A.F, *B = A.B;
    if (s.stage) {
        int off = 0;
        for (int e = 0; e < a; ++e) off += 2 * s.ax[e].n * s.ax[e].hp;
        F = mats + off;
        B = F + n * A.hp;
    }
    double mine = 0.0;
    for (int L0 = blockIdx.x * nl; L0 < lines; L0 += gridDim.x * nl)
        mine = small_axis<MODE>(A, F, B, work, work + nl * n, sr, in, out, tag, scale, inner, L0,
                                lines - L0 < nl ? lines - L0 : nl, tl, nb, wt);
    return mine;
}

// The solve's correction to the warm start, (I - g L)^{-1} r.
__device__ __forceinline__ double small_dct(const MeshDev& m, const SmallArgs& s, int i, int slot, int p, bool has, int tl,
                                            int nb, double r, double* mats, double* work, SmallWait& wt)
{
    const double* scale = s.winv + (size_t)(i - 1) * m.ld;
    const SmallTag tag = slot + 1;
    const int N = m.N;
    auto buf = [&](int b) { return s.cells + (size_t)b * N; };
    // whole x lines lie in their own block's nodes when nx divides the block
    const bool local = m.nx > 1 && nb % m.nx == 0;
    double* sr = work + 2 * (nb > 1 ? nb : 1);
    if (local) {
        sr[tl] = has ? r : 0.0;
        v_sync(nb);
    } else if (has) {
        cell_put(buf(kBufR) + p, r, tag);
    }
    const int last = m.nz > 1 ? 2 : (m.ny > 1 ? 1 : 0);
    const SmallCell* in = local ? nullptr : buf(kBufR);
    double e = 0.0;
    bool own = false;                            // e is already the thread's own node's
    if (last == 0) {
        e = small_axis_all<2>(s, m, 0, mats, work, sr, in, local ? nullptr : buf(kBufE), tag, scale, tl, nb, wt);
        own = local;
    } else {
        if (m.nx > 1) {
            small_axis_all<0>(s, m, 0, mats, work, sr, in, buf(kBufX), tag, nullptr, tl, nb, wt);
            in = buf(kBufX);
        }
        const bool ymid = last == 2 && m.ny > 1;
        if (ymid) {
            small_axis_all<0>(s, m, 1, mats, work, nullptr, in, buf(kBufY), tag, nullptr, tl, nb, wt);
            in = buf(kBufY);
        }
        small_axis_all<2>(s, m, last, mats, work, nullptr, in, buf(m.nx > 1 || ymid ? kBufZ : kBufE), tag, scale, tl, nb, wt);
        in = buf(kBufZ);
        if (ymid) {
            small_axis_all<1>(s, m, 1, mats, work, nullptr, in, buf(m.nx > 1 ? kBufW : kBufE), tag, nullptr, tl, nb, wt);
            in = buf(kBufW);
        }
        if (m.nx > 1) {
            e = small_axis_all<1>(s, m, 0, mats, work, nullptr, in, local ? nullptr : buf(kBufE), tag, nullptr, tl, nb, wt);
            own = local;
        }
    }
    if (!own && has) e = cell_get(buf(kBufE), p, tag, wt);
    if (blockIdx.x == 0 && tl == 0) {
        s.status[0] = 1;
        if (slot < s.log_len) s.log[slot] = 1;
    }
    return e;
}

template <class Model, int M>
__global__ void __launch_bounds__(512, 1) k_small_step(const __grid_constant__ StepArgs a, const __grid_constant__ SmallArgs s)
{
    extern __shared__ double small_smem[];
    __shared__ double sV[2][512];                        // V of the last solves, for the gates' warps
    constexpr int NS = Model::NS, NA = Model::NA, NG = Model::NG;
    const MeshDev& m = a.m;
    const int64_t row = (int64_t)NS * m.ld, ld = m.ld;
    const int nb = 1 << s.lgnb, R = s.roles;
    const int role = threadIdx.x >> s.lgnb, tl = threadIdx.x & (nb - 1);
    const int p = blockIdx.x * nb + tl, N = m.N;
    const bool has = p < N;
    // gates [g0, g1) belong to this thread's role
    const int gper = R == 1 ? NG : (NG + R - 2) / (R - 1);
    const int g0 = R == 1 ? 0 : (role == 0 ? NG : min(NG, (role - 1) * gper)), g1 = role == 0 && R > 1 ? NG : min(NG, g0 + gper);
    NodeIdx n{0, 0, 0};
    if (has) n = node_idx(m, p);
    unsigned target = 0;
    SmallWait wt{s.bar, a.flags, false};
    double* mats = small_smem;
    double* work = small_smem + s.stage;
    // clear the cells' tags; the grid barrier below orders that before any use
    if (role == 0 && has)
        for (int b = 0; b < (s.dct ? (int)ESDC_SMALL_BUFS : 2); ++b) cell_put(s.cells + (size_t)b * N + p, 0.0, 0);
    if (threadIdx.x < 4) cell_put(s.part + (size_t)threadIdx.x * gridDim.x + blockIdx.x, 0.0, 0);
    SmallStencil st;
    if (role == 0) small_stencil(m, p, has, n, st);
    if (s.dct) {
        if (s.stage) {
            int off = 0;
            for (int e = 0; e < 3; ++e) {
                const int cnt = s.ax[e].n > 1 ? s.ax[e].n * s.ax[e].hp : 0;
                for (int w = threadIdx.x; w < cnt; w += blockDim.x) {
                    mats[off + w] = __ldg(s.ax[e].F + w);
                    mats[off + cnt + w] = __ldg(s.ax[e].B + w);
                }
                off += 2 * s.ax[e].n * s.ax[e].hp;
            }
        }
        if (has && role == R - 1) {
            const double mu = (s.ex[n.ix] + s.ey[n.iy]) + s.ez[n.iz];
#pragma unroll 1
            for (int i = 1; i <= M; ++i)
                __stcg(s.winv + (size_t)(i - 1) * ld + p, s.wgt * esdc::esdc_rcp(fma(-s.g[i], mu, 1.0)));
        }
    }
    NodeSolve so{0.0, 0.0, 0.0};
    double V = 0.0, Vn = 0.0;                            // V_{i-1}^{k+1}, V_n
    const float uf[NS] = {};
    double* Gold = s.G0;
    double* Gnew = s.G1;
    if (has) {
        Vn = V = a.yn[p];
        const PhaseArgs p0{0, 0.0, s.G0, s.G0, nullptr}, p1{1, 0.0, s.G0, s.G0, nullptr};
        const bool one = M >= 2 && s.fuse1;
        if (role == 0) {
            double u[NS];
#pragma unroll
            for (int e = 0; e < NS; ++e) u[e] = a.yn[e * ld + p];
            setup_v<Model, M, false>(a, p0, a.st, a.stim_on, a.D, lap(m, a.yn, p, n.ix, n.iy, n.iz), u, uf, p, n.ix, n.iy,
                                     n.iz);
            if (one)
                node_v<Model, M, false, false, true>(a, p1, a.st, a.stim_on, a.D, []() { return 0.0; }, u, uf, p, n.ix,
                                                     n.iy, n.iz, &so);
        }
        const typename Model::VCtx vc = Model::vctx(a.mp, V);
#pragma unroll 1
        for (int g = g0; g < g1; ++g) {
            setup_gate<Model, M, false>(a, p0, g, V, 0.0f, vc, p);
            if (one) node_gate<Model, M, false, false>(a, p1, g, a.yn[(1 + NA + g) * ld + p], V, 0.0f, vc, p);
        }
    }
    if (!grid_barrier(s.bar, target, a.flags)) wt.dead = true;
    SmallTag tag = 0, nred = 0;
    int slot = 0;
    for (int k = 0; k < s.K; ++k) {
#pragma unroll 1
        for (int i = 1; i <= M + 1; ++i) {
            const bool fused = M >= 2 && s.fuse1;
            if (has && !(fused && i == 1)) {
                const double rho = (i >= 2 && i <= M) ? (k == 0 ? s.rho0[i] : 1.0) : 0.0;
                // the second pass, when there is one, is node 1 of sweep k + 1
                const int passes = fused && i == M + 1 && k + 1 < s.K ? 2 : 1;
#pragma unroll 1
                for (int e = 0; e < passes; ++e) {
                    const PhaseArgs ph = e ? PhaseArgs{1, 0.0, Gnew, Gnew, nullptr} : PhaseArgs{i, rho, Gold, Gnew, nullptr};
                    const double* src = ph.i >= 2 ? a.Y + (int64_t)(ph.i - 2) * row : a.yn;
                    const double v = ph.i >= 2 ? V : Vn;
                    if (role == 0) {
                        double u[NS];
                        u[0] = v;
#pragma unroll
                        for (int q = 1; q < NS; ++q) u[q] = src[q * ld + p];
                        const SmallCell* vc = s.cells + (size_t)(s.dct ? (int)kBufV : (int)(tag & 1)) * N;
                        node_v<Model, M, false, false, true>(
                            a, ph, a.st, a.stim_on, a.D, [&]() { return small_lap(st, vc, s.dct ? (SmallTag)slot : tag, v, wt); },
                            u, uf, p, n.ix, n.iy, n.iz, &so);
                    }
                    if (g0 < g1) {
                        typename Model::VCtx vc{};
                        if (ph.i >= 2) vc = Model::vctx(a.mp, v);
#pragma unroll 1
                        for (int g = g0; g < g1; ++g)
                            node_gate<Model, M, false, false>(a, ph, g, src[(1 + NA + g) * ld + p], v, 0.0f, vc, p);
                    }
                }
            }
            if (i > M) {
                // With one node y_M is y_1: the gates' warps may write node 1 of the next sweep only after
                // the V warps have read y_1 for this evaluation.  (With more nodes that is another row, and
                // the barrier after its solve orders the rest.)
                if (M == 1 && k + 1 < s.K) __syncthreads();
                break;
            }
            if (role == 0) {
                double e;
                if (s.dct) e = small_dct(m, s, i, slot, p, has, tl, nb, so.r, mats, work, wt);
                else if (s.fourth) e = small_cheb<12>(st, s, N, i, slot, p, has, tl, nb, so, tag, nred, wt);
                else if (s.layers) e = small_cheb<10>(st, s, N, i, slot, p, has, tl, nb, so, tag, nred, wt);
                else e = small_cheb<6>(st, s, N, i, slot, p, has, tl, nb, so, tag, nred, wt);
                if (has) {
                    V = so.x + e;
                    a.Y[(int64_t)(i - 1) * row + p] = V;
                    if (s.dct) {
                        cell_put(s.cells + (size_t)kBufV * N + p, V, slot + 1);
                        if (!isfinite(V)) atomicOr(a.flags, ESDC_FLAG_NONFINITE);
                    } else {
                        cell_put(s.cells + (size_t)((tag + 1) & 1) * N + p, V, tag + 1);
                    }
                    if (R > 1) sV[slot & 1][tl] = V;
                }
                ++tag;
            }
            __syncthreads();                             // V_i for the gates' warps, y_i's gates for the V warps
            if (role > 0 && has) V = sV[slot & 1][tl];
            ++slot;
        }
        double* t = Gold; Gold = Gnew; Gnew = t;
    }
    // residual and output: this node's values only, the states shared out over the roles
    __shared__ unsigned long long smax[2 * ESDC_NSMAX];
    for (int e = threadIdx.x; e < 2 * NS; e += blockDim.x) smax[e] = 0ULL;
    __syncthreads();
    bool bad = false;
    if (has) {
#pragma unroll 1
        for (int e = role; e < NS; e += R) {
            double rmax = 0.0, ymax = 0.0;
            bad |= !residual_state<Model, M>(a, PhaseArgs{0, 0.0, Gold, nullptr, s.yout}, p, e, rmax, ymax);
            atomicMax(&smax[e], (unsigned long long)__double_as_longlong(rmax));
            atomicMax(&smax[NS + e], (unsigned long long)__double_as_longlong(ymax));
        }
    }
    if (bad) atomicOr(a.flags, ESDC_FLAG_NONFINITE);
    __syncthreads();
    for (int e = threadIdx.x; e < 2 * NS; e += blockDim.x) atomicMax(a.rmax + e, smax[e]);
}

template <class Model, int M>
cudaError_t small_launch(const StepArgs& a, const SmallArgs& s, int blocks, int threads, size_t smem, cudaStream_t st)
{
    const void* k = (const void*)k_small_step<Model, M>;
    // The opt-in to more than 48 KB of shared memory (which the kernel's own arrays count towards), once per kernel
    // and device and for the largest step, so that no other thread's smaller mesh takes it back before the launch.
    static std::atomic<unsigned long long> opted{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ULL << (dev & 63);
    if (smem > 0 && (dev > 63 || !(opted.load(std::memory_order_acquire) & bit))) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(double) * (kSmallStageDoubles + 3 * 512)));
        if (e != cudaSuccess) return e;
        opted.fetch_or(bit, std::memory_order_release);
    }
    void* args[] = {const_cast<StepArgs*>(&a), const_cast<SmallArgs*>(&s)};
    return cudaLaunchCooperativeKernel(k, dim3(blocks), dim3(threads), args, smem, st);
}

template <class Model>
cudaError_t small_launch_M(const StepArgs& a, const SmallArgs& s, int M, int blocks, int threads, size_t smem,
                           cudaStream_t st)
{
    switch (M) {
        case 1: return small_launch<Model, 1>(a, s, blocks, threads, smem, st);
        case 2: return small_launch<Model, 2>(a, s, blocks, threads, smem, st);
        case 3: return small_launch<Model, 3>(a, s, blocks, threads, smem, st);
        case 4: return small_launch<Model, 4>(a, s, blocks, threads, smem, st);
        case 5: return small_launch<Model, 5>(a, s, blocks, threads, smem, st);
        case 6: return small_launch<Model, 6>(a, s, blocks, threads, smem, st);
        case 7: return small_launch<Model, 7>(a, s, blocks, threads, smem, st);
        case 8: return small_launch<Model, 8>(a, s, blocks, threads, smem, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace
