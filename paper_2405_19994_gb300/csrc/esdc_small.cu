// One-launch steps of small meshes: the choice, the tables and the Hodgkin-Huxley
// model's kernels (esdc_small.cuh holds the device side).
#include <mutex>

#include "esdc_small.cuh"

namespace {

std::mutex g_const_mu;
bool g_const_done[64] = {false};

// Nodes per block up to which a step runs as one launch (N <= SMs times that).
// One launch against the sequence with k_small_solve (us per step, HH M = 3 K = 4 /
// SYN19 M = 4 K = 6): scalar sheets of 7,575 nodes 332 / 435 and 859 / 1324, 21,000 462 /
// 492 and 1263 / 1500, 38,805 494 / 548 and 1564 / 1918; above the line (512 nodes per
// block, one role, 16 warps' FP64 issue) 42,000 nodes 846 / 634, 77,000 939 / 706, SYN19
// 65,536 2923 / 2412.  The line is late for what has more neighbours: 37,800 layered nodes
// 616 / 609 (SYN19 1941 / 2079), 38,805 of the fourth order 745 / 652.
// Fields have a line of their own from when the sequence solved them with k_cheb (65,536
// nodes 1084 / 1288); with k_small_solve the sequence is the faster one above 256 nodes
// per SM for them too: 42,000 nodes 940 / 711, 65,536 974 / 767 and SYN19 3287 / 2690.
constexpr int kSmallNodes = 256, kSmallNodesField = 512;
// Dense cosine products against the sequence's FFT passes: N sum(n + 2) FP64
// operations per solve over two lanes per SM and clock (us per step, HH / SYN19 as
// above).  128x128 (14,000 cycles) 587 against 696 and 1239 / 1779, 64x32x16 (12,500) 445 / 700,
// 256x64 (17,500) 710 / 672 and 1664 / 1728; above the line 256x128 (42,000) 802 / 746 and
// 2360 / 2170; 256x256 would be 111,000 cycles, four times the FFT solve.
constexpr double kSmallDctCycles = 40000.0;
constexpr int kSmallDctAxis = 256;
constexpr int kSmallDctCable = 128;         // 1D: one line means one block

bool dct_small(const esdc_handle* h)
{
    const int n[3] = {h->mesh.nx, h->mesh.ny, h->mesh.nz};
    double ops = 0.0;
    int axes = 0, last = 1;
    for (int a = 0; a < 3; ++a) {
        if (n[a] == 1) continue;
        if (n[a] > kSmallDctAxis) return false;
        ops += n[a] + 2.0;
        ++axes;
        last = n[a];
    }
    if (axes == 0 || (axes < 2 && last > kSmallDctCable)) return false;
    return ops * h->mesh.N / (2.0 * h->sms) <= kSmallDctCycles;
}

// One Chebyshev solve by itself: the semi-iteration of the one-launch step (small_cheb) on the
// correction to the guess x, for meshes of up to a node per thread of one 512-thread block per SM.
// The launch sequences of such meshes (the adjoint's, and those above kSmallNodes) ran k_cheb or
// k_cheb4, whose iteration is a store, a grid barrier and a load: 86 us per solve of the 256x256
// field sheet, 48 here (an iteration is bound by the 16 warps' FP64 issue).  Tags go on from
// launch to launch (the cells need no clearing, so there is no barrier): every block
// takes the first from device memory, and block 0 moves it on when the solve has ended,
// after every block has posted a sum under it.
struct SolveArgs {
    MeshDev m;
    int maxit, log_len;
    double tol2;
    const double* b;
    double* x;
    SmallCell *cells, *part;
    unsigned long long* tag;
    unsigned long long stride;       // tags a solve may use
    unsigned* bar;
    int *status, *log, *flags;
    double g[1], inv_theta[1], log_q;
    double ca[1][ESDC_SMALL_TAB], cb[1][ESDC_SMALL_TAB], qq[1][ESDC_SMALL_TAB];
};

template <int NB>
__global__ void __launch_bounds__(512, 1) k_small_solve(const __grid_constant__ SolveArgs s)
{
    const MeshDev& m = s.m;
    const int nb = blockDim.x, tl = threadIdx.x, p = blockIdx.x * nb + tl, N = m.N;
    const bool has = p < N;
    const SmallTag tag0 = __ldcg(s.tag);
    SmallStencil st;
    small_stencil(m, p, has, has ? node_idx(m, p) : NodeIdx{0, 0, 0}, st);
    NodeSolve so{0.0, 0.0, 0.0};
    if (has) {
        so.b = s.b[p];
        so.x = s.x[p];
        double t = 0.0;
#pragma unroll
        for (int e = 0; e < NB; ++e)
            if ((st.mask >> e) & 1u) t = fma(st.cf[e], s.x[st.q[e]] - so.x, t);
        so.r = fma(s.g[0], t, so.b - so.x);
    }
    SmallTag tag = tag0, nred = tag0;
    SmallWait wt{s.bar, s.flags, false};
    const bool mute = __ldcg(s.bar + 2) == blockIdx.x + 1;
    const double e = small_cheb<NB, true>(st, s, N, 0, 0, p, has, tl, nb, so, tag, nred, wt, mute);
    // every block has posted its first sum, so every neighbour has read its x
    if (has) s.x[p] = so.x + e;
    if (blockIdx.x == 0 && tl == 0) *s.tag = tag0 + s.stride;
}

}  // namespace

cudaError_t esdc_small_solve(const MeshDev& m, const CgWork& w, double g, const ChebArgs& c, const double* b, double* x,
                             double tol, int maxit, int* iter_log, int* flags, cudaStream_t st)
{
    SolveArgs s;
    s.m = m;
    s.maxit = maxit;
    s.log_len = iter_log ? 1 : 0;
    s.tol2 = tol * tol;
    s.b = b;
    s.x = x;
    s.cells = static_cast<SmallCell*>(w.cells);
    s.part = static_cast<SmallCell*>(w.cell_part);
    s.tag = w.cell_tag;
    s.stride = 2ULL * (unsigned)maxit + 64;
    s.bar = w.bar;
    s.status = w.status;
    s.log = iter_log;
    s.flags = flags;
    s.g[0] = g;
    s.inv_theta[0] = c.inv_theta;
    s.log_q = c.log_q;
    double q2 = 1.0;
    for (int k = 0; k < ESDC_SMALL_TAB; ++k) {
        s.ca[0][k] = c.ca[k];
        s.cb[0][k] = c.cb[k];
        q2 *= c.q * c.q;
        s.qq[0][k] = 4.0 * q2;
    }
    int nodes = 32;
    while ((m.N + nodes - 1) / nodes > w.sms) nodes *= 2;
    const void* k = m.order == 4 ? (const void*)k_small_solve<12>
                  : m.lay ? (const void*)k_small_solve<10> : (const void*)k_small_solve<6>;
    void* args[] = {&s};
    return cudaLaunchCooperativeKernel(k, dim3((m.N + nodes - 1) / nodes), dim3(nodes), args, 0, st);
}

cudaError_t esdc_small_launch_hh(const StepArgs& a, const void* args, int M, int blocks, int threads, size_t smem,
                                 cudaStream_t s)
{
    return small_launch_M<esdc::HH1952>(a, *static_cast<const SmallArgs*>(args), M, blocks, threads, smem, s);
}

cudaError_t esdc_small_prepare(esdc_handle* h)
{
    SmallDev& d = h->small;
    d = SmallDev{};
    if (h->opt.precision != 0 || h->opt.solver == 1 || (long long)h->mesh.N > (long long)h->sms * kSmallNodesField)
        return cudaSuccess;
    cudaError_t e;
    if (h->model == ESDC_MODEL_HH1952) {
        std::lock_guard<std::mutex> lk(g_const_mu);
        e = upload_constants_local(g_const_done, h->device);
    } else {
        e = esdc_small_constants_syn(h->device);
    }
    if (e != cudaSuccess) return e;
    const bool dct = h->cg.dct && dct_small(h);
    e = cudaMalloc(&d.part, sizeof(SmallCell) * 4 * h->sms);
    if (e != cudaSuccess) return e;
    if ((e = cudaMalloc(&d.cells, sizeof(SmallCell) * (dct ? (int)ESDC_SMALL_BUFS : 2) * h->mesh.N)) != cudaSuccess) return e;
    // tags of the solves start above any that a step's launch uses
    const unsigned long long tag0 = 1ULL << 40;
    if ((e = cudaMalloc((void**)&d.tag, sizeof tag0)) != cudaSuccess) return e;
    if ((e = cudaMemcpy(d.tag, &tag0, sizeof tag0, cudaMemcpyHostToDevice)) != cudaSuccess) return e;
    if ((e = cudaMemset(d.cells, 0, sizeof(SmallCell) * 2 * h->mesh.N)) != cudaSuccess) return e;
    if ((e = cudaMemset(d.part, 0, sizeof(SmallCell) * 4 * h->sms)) != cudaSuccess) return e;
    h->cg.cells = d.cells;
    h->cg.cell_part = d.part;
    h->cg.cell_tag = d.tag;
    h->cg.cell_nodes = h->sms * kSmallNodesField;
    h->cg.sms = h->sms;
    if (!dct) return cudaSuccess;
    const int n[3] = {h->mesh.nx, h->mesh.ny, h->mesh.nz};
    std::vector<double> mats;
    size_t off[3] = {0, 0, 0};
    for (int a = 0; a < 3; ++a) {
        const int na = n[a], hp = (na + 1) / 2;
        d.ax[a].n = na;
        d.ax[a].hp = hp;
        off[a] = mats.size();
        mats.resize(mats.size() + 2 * (size_t)na * hp, 0.0);
        double* F = mats.data() + off[a];
        double* B = F + (size_t)na * hp;
        // k (2 i + 1) is reduced modulo 4 n as an integer: the argument of the cosine stays below 2 pi
        for (int i = 0; i < hp; ++i)
            for (int k = 0; k < na; ++k) {
                const long long q = (long long)k * (2 * i + 1) % (4LL * na);
                const double c = std::cos(M_PI * (double)q / (2.0 * na));
                F[(size_t)i * na + k] = c;
                B[(size_t)k * hp + i] = (k == 0 ? 1.0 : 2.0) * c;
            }
    }
    if ((e = cudaMalloc((void**)&d.winv, sizeof(double) * h->opt.M_max * h->mesh.ld)) != cudaSuccess) return e;
    if ((e = cudaMalloc((void**)&d.mats, sizeof(double) * mats.size())) != cudaSuccess) return e;
    if ((e = cudaMemcpy(d.mats, mats.data(), sizeof(double) * mats.size(), cudaMemcpyHostToDevice)) != cudaSuccess)
        return e;
    for (int a = 0; a < 3; ++a) {
        d.ax[a].F = d.mats + off[a];
        d.ax[a].B = d.ax[a].F + (size_t)n[a] * d.ax[a].hp;
    }
    d.mat_doubles = (int)mats.size();
    return cudaSuccess;
}

void esdc_small_destroy(SmallDev* d)
{
    void* ptrs[] = {d->part, d->cells, d->mats, d->winv, d->tag};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    *d = SmallDev{};
}

cudaError_t esdc_small_step(esdc_handle* h, StepArgs& a, double* y, int M, int K, cudaStream_t st, bool* taken)
{
    *taken = false;
    const SmallDev& d = h->small;
    // the adjoint's recording copies the iterate between sweeps: launch sequence
    if (!d.part || K < 1 || h->tapeY) return cudaSuccess;
    int solver = 0;
    if (esdc_get_solver(h, &solver) != ESDC_OK) return cudaSuccess;
    const ColloData* C = &h->col[M - 1];
    SmallArgs s;
    s.dct = solver == 2;
    if (s.dct && !d.mats) return cudaSuccess;
    if ((long long)h->mesh.N > (long long)h->sms * (h->mesh.sig ? kSmallNodesField : kSmallNodes)) return cudaSuccess;
    for (int i = 1; i <= M; ++i) {
        s.g[i] = a.dt * C->d[i] * h->D;
        s.rho0[i] = i >= 2 ? C->c[i] / C->c[i - 1] : 0.0;
        s.inv_theta[i] = 0.0;
        if (!(s.g[i] > 0.0)) return cudaSuccess;
        if (s.dct) continue;
        ChebArgs c;
        if (!esdc_cheb_interval(h->mesh, s.g[i], c)) return cudaSuccess;
        s.inv_theta[i] = c.inv_theta;
        double q2 = 1.0;
        for (int k = 0; k < ESDC_SMALL_TAB; ++k) {
            s.ca[i][k] = c.ca[k];
            s.cb[i][k] = c.cb[k];
            q2 *= c.q * c.q;
            s.qq[i][k] = 4.0 * q2;
        }
    }
    s.g[0] = s.rho0[0] = s.inv_theta[0] = 0.0;
    s.layers = h->mesh.lay != nullptr;
    s.fourth = h->mesh.order == 4;
    s.K = K;
    s.fuse1 = h->opt.fuse_node1 && M >= 2;
    s.maxit = h->opt.cg_maxit;
    s.tol2 = h->opt.tol_cg * h->opt.tol_cg;
    s.G0 = h->G0; s.G1 = h->G1; s.yout = y;
    s.cells = static_cast<SmallCell*>(d.cells);
    s.part = static_cast<SmallCell*>(d.part);
    s.bar = h->cg.bar;
    s.status = h->cg.status;
    s.log = h->cg_log; s.log_len = h->cg_log_len;
    s.stage = 0;
    s.winv = d.winv;
    s.ex = h->dct.ex; s.ey = h->dct.ey; s.ez = h->dct.ez;
    s.wgt = 1.0;
    // The fewest nodes per block that give every node a thread on some SM: the
    // FP64 work spreads over as many SMs as there are warps.  Blocks of up to 128
    // nodes split a node over four roles and of 256 over two (512 threads at most).
    const int N = h->mesh.N;
    int nodes = 32;
    while ((N + nodes - 1) / nodes > h->sms) nodes *= 2;
    size_t smem = 0;
    if (s.dct) {
        int longest = 1;
        for (int e = 0; e < 3; ++e) {
            s.ax[e] = d.ax[e];
            if (d.ax[e].n > longest) longest = d.ax[e].n;
            if (d.ax[e].n > 1) s.wgt /= d.ax[e].n;
        }
        while (nodes < longest) nodes *= 2;                                     // a line's outputs in one pass
        if (d.mat_doubles <= kSmallStageDoubles) s.stage = d.mat_doubles;
        smem = sizeof(double) * ((size_t)s.stage + 3 * (size_t)nodes);
    }
    s.roles = nodes <= 128 ? 4 : (nodes == 256 ? 2 : 1);
    s.lgnb = 0;
    while ((1 << s.lgnb) < nodes) ++s.lgnb;
    const int threads = nodes * s.roles, blocks = (N + nodes - 1) / nodes;
    step_constants(h, a, M);
    a.ztab = esdc_ztab_device(h->zt, M, a.dt, *C, st);
    prof_begin(h, 1, st);
    const cudaError_t e = h->model == ESDC_MODEL_HH1952 ? esdc_small_launch_hh(a, &s, M, blocks, threads, smem, st)
                                                         : esdc_small_launch_syn(a, &s, M, blocks, threads, smem, st);
    prof_end(h, st);
    if (e == cudaSuccess) {
        *taken = true;
        h->last_Gfinal = (K & 1) ? h->G1 : h->G0;
    }
    return e;
}
