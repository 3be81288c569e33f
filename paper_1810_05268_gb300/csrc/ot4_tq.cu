// OT4 steps fed by tensor copies (3D, Tile.ver 10): the passes of ot4.cu on
// the ring, queue and tile of the tensor-copy OT2 kernels (stencil_tq.cu).
//
// The vector-blocked passes (ot4_v3.cu) load a plane by every thread's own
// vectors and keep them, a plane ahead, in registers: 166 registers, three
// CTAs an SM, and the passes that stage two fields hold two queues.  Here one
// thread issues a plane's copies (the halo'd tile of the staged field and a
// point tile of each other field), the others wait on the plane's mbarrier,
// and every pass stages one field, so five CTAs fit an SM.  The reverse step
// is four passes instead of three:
//   1. stages lam^j:     Z_l = w lap, and the deferred g += Z_u(j+1) lap / 12
//   2. stages Z_l:       lam^{j-1} by the update (the forward step's pass 2)
//   3. stages u^{j-1}:   Z_u(j) = w lap, and lap itself (over Z_l's field)
//   4. stages Z_u(j):    g += lam^{j-1} (lap u^{j-1} + lap Z_u / 12 + q)
// which moves 80 B/pt against 72 for three passes of two staged fields, and
// the forward step 12 + 20 as before.  At 208^3, order 8: forward 92 -> 71 us,
// reverse 205 -> 145 us a step (4.1 and 5.0 TB/s of the passes' own traffic).
// The operations and their order are the
// other generations', so the results are bitwise theirs.
#include "tq_common.cuh"

namespace ckfwi {
namespace {

enum { OP_LAP, OP_LAP_LAM, OP_LAP_U, OP_UPDATE, OP_GRAD };

// point fields of a pass, in the order of its maps
constexpr int points_of(int op)
{
    return op == OP_LAP || op == OP_LAP_U ? 1 : 3;   // w | w, Z_u(j+1), g | w | f, previous f, w | lap u, lam^{j-1}, g
}

template <int NP>
struct Maps4 {
    CUtensorMap f, p[NP];
};

// CTAs an SM at order <= 8: shared memory and registers of one point field
// allow one more than those of three
template <int K, int PF, int OP> constexpr int ot4q_min_blocks() { return K > 4 ? (PF == 1 ? 4 : 3) : (points_of(OP) == 1 ? 7 : 6) - PF; }

template <int K, int PF, int OP, int CK>
__global__ void __launch_bounds__(128, ot4q_min_blocks<K, PF, OP>())
    ot4q_kernel(const Ot4qArgs A, const __grid_constant__ Maps4<points_of(OP)> M)
{
    constexpr int NP = points_of(OP);
    using Q = TQ<K, PF, NP>;
    using G = typename Q::G;
    constexpr int V = Q::V, TX = Q::TX, TY = Q::TY, D = Q::D, RU = Q::RU, RP = Q::RP, LD = Q::LEAD;
    extern __shared__ unsigned char smq_raw[];
    __shared__ int abort_s[2];                  // a wait gave up at a step of this parity
    unsigned char* sm0 = align128(smq_raw);
    float* ring = reinterpret_cast<float*>(sm0);
    float* pts = ring + RU * Q::US;             // field k, slot s: pts + (k * RP + s) * PT
    uint64_t* bar = reinterpret_cast<uint64_t*>(pts + NP * RP * Q::PT);
    const FwdArgs& a = A.f;

    const int bxi = blockIdx.x, byi = blockIdx.y, bzi = blockIdx.z;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int nz = a.g.nz, ny = a.g.ny, nx = a.g.nx;
    const int px = (int)a.g.px, pxy = (int)a.g.pxy;
    const int xb = bxi * G::BXP, yb = byi * TY;
    const int x0 = xb + V * tx;
    const int y = yb + ty;

    if (OP == OP_LAP && a.smp.n > 0) {   // receiver sampling of u^n by the first threads of the grid
        const int gt = ((bzi * gridDim.y + byi) * gridDim.x + bxi) * (TX * TY) + tid;
        if (gt < a.smp.n) {
            float acc = 0.0f;
            for (int i = 0; i < a.smp.nst; ++i)
                acc = __fmaf_rn(a.smp.wt[gt * a.smp.nst + i], __ldg(A.s + a.smp.idx[gt * a.smp.nst + i]), acc);
            a.smp.out[gt] = acc;
        }
    }

    const int z0 = bzi * a.zlen;
    if (z0 >= nz) return;                       // the whole CTA: no copy issued yet
    const int z1 = min(z0 + a.zlen, nz);
    const int nstep = z1 - z0;
    const bool rowact = y < ny;
    const bool cload = rowact && x0 < nx;
    const bool full = rowact && x0 + V <= nx;
    const int col = y * px + x0;
    const int cs = (ty + K) * G::RX + G::PX + V * tx;
    const int ps = ty * G::BXP + V * tx;
    float ecol[V];
    if (OP == OP_UPDATE) {
#pragma unroll
        for (int i = 0; i < V; ++i)
            ecol[i] = (rowact && x0 + i < nx) ? __fadd_rn(a.eta[nz + y], a.eta[nz + ny + x0 + i]) : 0.0f;
    }
    Inj3<V> ij;
    if (OP == OP_UPDATE || OP == OP_GRAD) ij.init(a.src, y, x0, nx, rowact);
    const int zqmax = nz + K - 1;
    const long long rounds = a.wait_limit;

    // copy group g: plane z0 + g of the staged field and, from g = K on, the
    // point planes z0 + g - K (see stencil_tq.cu)
    auto issue = [&](int g) {
        uint64_t* b = bar + g % RU;
        const bool pt = g >= LD;
        bar_expect(b, Q::UBYTES + (pt ? NP * Q::PBYTES : 0));
        tile3(ring + (g % RU) * Q::US, &M.f, xb, yb, min(z0 + g, zqmax) + K, b);
        if (pt) {
            const int zp = min(z0 + g - LD, z1 - 1) + K, s = (g - LD) % RP;
#pragma unroll
            for (int k = 0; k < NP; ++k) tile3(pts + (k * RP + s) * Q::PT, &M.p[k], xb + G::PX, yb + K, zp, b);
        }
    };
    auto wait_group = [&](int g) { return bar_wait(bar + g % RU, (unsigned)((g / RU) & 1), rounds); };

    if (tid == 0) {
        abort_s[0] = abort_s[1] = 0;
        for (int s = 0; s < RU; ++s) bar_init(bar + s);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int g = 0; g < LD + D; ++g) issue(g);
    }
    __syncthreads();
    int issued = LD + D;
    float q[2 * K + 1][V], nq[V];
#pragma unroll
    for (int i = 0; i < (Q::COL ? 2 * K : K); ++i) {
        if (cload) gld<V>(q[i], A.s + (z0 - K + i) * pxy + col);
        else vzero<V>(q[i]);
    }
    if constexpr (Q::COL) {
        if (cload) gld<V>(nq, A.s + (z0 + K) * pxy + col);
        else vzero<V>(nq);
    }
    int g0 = 0;
    while (g0 < LD && wait_group(g0)) ++g0;
    if (g0 < LD) abort_s[0] = 1;
    bool aborted = false;                        // the same in every thread: read after one barrier
    int confirmed = g0;
#pragma unroll
    for (int i = 0; i < LD; ++i) sld<V>(q[K + i], ring + i * Q::US + cs);

    for (int step = 0; step < nstep; ++step) {
        const int z = z0 + step;
        if (!wait_group(step + LD)) abort_s[step & 1] = 1;
        __syncthreads();                        // every thread is past step - 1: its slots are free
        if (abort_s[step & 1]) {
            aborted = true;
            break;
        }
        confirmed = step + LD + 1;
        if (tid == 0) issue(step + LD + D);
        issued = step + LD + D + 1;
        if constexpr (Q::COL) {
#pragma unroll
            for (int k = 0; k < V; ++k) q[2 * K][k] = nq[k];
            if (cload) gld<V>(nq, A.s + min(z + K + 1, zqmax) * pxy + col);
        } else {
            sld<V>(q[2 * K], ring + ((step + K) % RU) * Q::US + cs);
        }
        const float* sm = ring + (step % RU) * Q::US;
        if (cload) {
            float pv[NP][V], r[V], l[V];
#pragma unroll
            for (int k = 0; k < NP; ++k) sld<V>(pv[k], pts + (k * RP + step % RP) * Q::PT + ps);
            const long long o = (long long)z * pxy + col;
            if (OP == OP_LAP || OP == OP_LAP_LAM || OP == OP_LAP_U) {
                lap3<K, V, TX, TY>(l, q, sm, tx, ty, a.c);
                if (OP == OP_LAP_U) vput<V>(A.lap, o, l, full, x0, nx);
#pragma unroll
                for (int p = 0; p < V / 2; ++p) {
                    const float2 t = __fmul2_rn(f2(pv[0][2 * p], pv[0][2 * p + 1]), f2(l[2 * p], l[2 * p + 1]));
                    r[2 * p] = t.x;
                    r[2 * p + 1] = t.y;
                }
                vput<V>(a.out, o, r, full, x0, nx);
            }
            if constexpr (OP == OP_LAP_LAM) {
                lap3<K, V, TX, TY>(l, q, sm, tx, ty, A.c12);
#pragma unroll
                for (int p = 0; p < V / 2; ++p) {
                    const float2 t = __ffma2_rn(f2(pv[1][2 * p], pv[1][2 * p + 1]), f2(l[2 * p], l[2 * p + 1]),
                                                f2(pv[2][2 * p], pv[2][2 * p + 1]));
                    r[2 * p] = t.x;
                    r[2 * p + 1] = t.y;
                }
                vput<V>(A.gacc, o, r, full, x0, nx);
            }
            if constexpr (OP == OP_UPDATE) {
                lap3<K, V, TX, TY>(l, q, sm, tx, ty, A.c12);
                ij.add(l, a.src, z);
                const float ez = a.eta[z];
                const float* zc = q[K];
#pragma unroll
                for (int p = 0; p < V / 2; ++p) {
                    const int i = 2 * p;
                    const float2 eta = __fadd2_rn(f2(ez, ez), f2(ecol[i], ecol[i + 1]));
                    const float2 t = leap4v(f2(pv[0][i], pv[0][i + 1]), f2(pv[1][i], pv[1][i + 1]), f2(pv[2][i], pv[2][i + 1]),
                                            f2(zc[i], zc[i + 1]), f2(l[i], l[i + 1]), eta, a.hdt);
                    r[i] = t.x;
                    r[i + 1] = t.y;
                }
                vput<V>(a.out, o, r, full, x0, nx);
                if (CK == CK_FP32) {
                    vput<V>(static_cast<float*>(a.ck_up), o, pv[0], full, x0, nx);
                } else if (CK == CK_BF16) {
                    st16<__nv_bfloat16, V>(a.ck_u, o, r, full, x0, nx);
                    st16<__nv_bfloat16, V>(a.ck_up, o, pv[0], full, x0, nx);
                } else if (CK == CK_FP16) {
                    const bool inf = st16<__half, V>(a.ck_u, o, r, full, x0, nx) | st16<__half, V>(a.ck_up, o, pv[0], full, x0, nx);
                    if (inf) atomicOr(a.err, 1);
                }
            }
            if constexpr (OP == OP_GRAD) {
                lap3<K, V, TX, TY>(l, q, sm, tx, ty, A.c12);
#pragma unroll
                for (int p = 0; p < V / 2; ++p) {
                    const float2 t = __fadd2_rn(f2(pv[0][2 * p], pv[0][2 * p + 1]), f2(l[2 * p], l[2 * p + 1]));
                    l[2 * p] = t.x;
                    l[2 * p + 1] = t.y;
                }
                ij.add(l, a.src, z);
#pragma unroll
                for (int p = 0; p < V / 2; ++p) {
                    const float2 t = __ffma2_rn(f2(pv[1][2 * p], pv[1][2 * p + 1]), f2(l[2 * p], l[2 * p + 1]),
                                                f2(pv[2][2 * p], pv[2][2 * p + 1]));
                    r[2 * p] = t.x;
                    r[2 * p + 1] = t.y;
                }
                vput<V>(A.gacc, o, r, full, x0, nx);
            }
        }
#pragma unroll
        for (int i = 0; i < 2 * K; ++i) {
#pragma unroll
            for (int k = 0; k < V; ++k) q[i][k] = q[i + 1][k];
        }
    }
    // no copy may land after the CTA has left (see stencil_tq.cu)
    if (tid == 0) {
        bool drained = true;
        for (int g = confirmed; g < issued; ++g)
            drained = bar_wait(bar + g % RU, (unsigned)((g / RU) & 1), DRAIN_ROUNDS) && drained;
        if (aborted || !drained) atomicOr(a.err, 8);
    }
}

template <int K, int PF, int OP, int CK>
cudaError_t op_go(const Ot4qArgs& A, const CUtensorMap* maps, cudaStream_t s)
{
    constexpr int NP = points_of(OP);
    using Q = TQ<K, PF, NP>;
    using G = typename Q::G;
    const FieldGeom& g = A.f.g;
    const dim3 blk(Q::TX, Q::TY, 1);
    const dim3 grd((g.nx + G::BXP - 1) / G::BXP, (g.ny + Q::TY - 1) / Q::TY, (g.nz + A.f.zlen - 1) / A.f.zlen);
    Maps4<NP> M;
    M.f = maps[0];
    for (int k = 0; k < NP; ++k) M.p[k] = maps[1 + k];
    cudaError_t e = cudaFuncSetAttribute(ot4q_kernel<K, PF, OP, CK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Q::SMEM);
    if (e != cudaSuccess) return e;
    ot4q_kernel<K, PF, OP, CK><<<grd, blk, Q::SMEM, s>>>(A, M);
    return cudaGetLastError();
}

template <int K, int PF>
cudaError_t op_k(int op, const Ot4qArgs& A, const CUtensorMap* maps, int ck, cudaStream_t s)
{
    switch (op) {
    case OT4Q_LAP: return op_go<K, PF, OP_LAP, CK_NONE>(A, maps, s);
    case OT4Q_LAP_LAM: return op_go<K, PF, OP_LAP_LAM, CK_NONE>(A, maps, s);
    case OT4Q_LAP_U: return op_go<K, PF, OP_LAP_U, CK_NONE>(A, maps, s);
    case OT4Q_GRAD: return op_go<K, PF, OP_GRAD, CK_NONE>(A, maps, s);
    case OT4Q_UPDATE:
        switch (ck) {
        case CK_NONE: return op_go<K, PF, OP_UPDATE, CK_NONE>(A, maps, s);
        case CK_FP32: return op_go<K, PF, OP_UPDATE, CK_FP32>(A, maps, s);
        case CK_BF16: return op_go<K, PF, OP_UPDATE, CK_BF16>(A, maps, s);
        case CK_FP16: return op_go<K, PF, OP_UPDATE, CK_FP16>(A, maps, s);
        default: return cudaErrorInvalidValue;
        }
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

bool ot4q_supported(int dims, int K, const Tile& t)
{
    return dims == 3 && t.ver == 10 && (K == 1 || K == 2 || K == 4 || K == 8) && t.bx == 32 && t.by == 16 &&
           t.vec == 4 && t.zlen >= 1 && (t.pf == 1 || t.pf == 2);
}

cudaError_t launch_ot4q(int op, const Ot4qArgs& A, const CUtensorMap* maps, const Tile& t, int K, int ck, cudaStream_t s)
{
    const FieldGeom& g = A.f.g;
    if (!v3_fits(g, K) || !ot4q_supported(g.dims, K, t)) return cudaErrorInvalidValue;
    // the boxes assume the first interior column at PX and H = K halo cells
    if (g.X0 != (K <= 4 ? 4 : 8) || g.H != K) return cudaErrorInvalidValue;
    Ot4qArgs B = A;
    B.f.zlen = t.zlen;
    switch (K) {
    case 1: return t.pf == 2 ? op_k<1, 2>(op, B, maps, ck, s) : op_k<1, 1>(op, B, maps, ck, s);
    case 2: return t.pf == 2 ? op_k<2, 2>(op, B, maps, ck, s) : op_k<2, 1>(op, B, maps, ck, s);
    case 4: return t.pf == 2 ? op_k<4, 2>(op, B, maps, ck, s) : op_k<4, 1>(op, B, maps, ck, s);
    case 8: return t.pf == 2 ? op_k<8, 2>(op, B, maps, ck, s) : op_k<8, 1>(op, B, maps, ck, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace ckfwi
