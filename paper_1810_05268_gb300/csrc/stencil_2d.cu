// 2D time steps, many per launch (Tile.ver 9): the forward step and the
// fused reverse step of the OT2 kernel with the whole grid held in the SMs'
// shared memory.
//
// A 2D field is small (464 x 1104: 2 MB, 281 x 281: 0.3 MB), so a step is
// bound by its launch and by the latency of one pass through the SMs, not by
// memory: one step per launch took 3.3 us (281 x 281, order 4) and 5.1 us
// (464 x 1104, order 8) of kernel time, 6.3 us launched from the host.  Here
// a launch advances up to STEP2_MAX steps.  The grid is cut into at most one
// tile per SM; a CTA keeps its bz x bx tile of u^n, u^{n-1} and w (and a K
// wide halo of u^n) in shared memory, and only the tiles' edges travel: each
// step half of a CTA's threads compute its edge points and publish them while
// the other half start on the interior, all share what is left of it, and the
// neighbours' edges become the next halo.  (Tiles that recompute their halos, several steps deep, so that CTAs
// never meet, were built first: 4.7 us a step at 464 x 1104, the redundant
// points cost more than the exchange.)
//
// Exchange.  A published vector of four values is two 16-byte stores of
// (value, epoch, value, epoch); the reader polls the data itself until every
// epoch is the one it waits for, so no fence or flag write is on the path.
// The epoch counts steps since the buffers were zeroed and is kept per tile
// in device memory (each CTA reads and writes only its own; a launch moves
// all by the same count), so a stale value never has the awaited epoch, also
// when a recorded graph is replayed.  Four buffers are used in turn: a CTA
// that writes step e needs its direct neighbours' step e - 1, hence every
// reader, the diagonal one too, has taken step e - 4.  The launch is
// cooperative (all tiles resident) and every wait is bounded: one that runs
// out raises error bit 8 and the CTA leaves at the end of the step; its
// neighbours' waits then run out as well.
//
// Edge points are computed by the first half of the threads, four x points
// each, interior points, the gradient's and the receivers by the threads
// after them, straight from shared memory: a row each while there are threads
// enough, else two rows at a time.  The arithmetic is lap_at's and leapfrog's, on pairs of
// points (packed FP32x2, each lane rounding like the scalar operation), so
// every value is bitwise the one the one-step kernels compute.  u^{n+1}
// overwrites u^{n-1} point by point.
//
// Measured, from set_model to the data on one GB300: 281 x 281, 500 steps
// 3.22 -> 0.95 ms (1.5 us a step, a reverse step 2.7); 464 x 1104, 2000 steps
// 12.5 -> 5.9 ms (2.9 and 4.8; lanes of a batch, whose tile is the least
// estimate's, 3.1 and 6.5).  What bounds it: a step's chain is an edge vector
// (about 1000 cycles: a lone warp issues an instruction every 6 cycles), the
// exchange (1350 cycles between two CTAs that do nothing else) and the
// interior beside it.  Two points a thread (1024 threads), all edges before
// any interior (a barrier between them) and the rare code out of line were
// each slower.
//
// What leaves a launch: the last two levels as the next state, any level that
// a checkpoint takes (FP32, BF16 or FP16: u^s of one checkpoint, u^{s-1} of
// the next), and the receivers of levels n .. n + T - 1, each by the tile
// that holds its first point (the other three are the tile's, or in its halo,
// whose one corner point is exchanged for this).
//
// The reverse step keeps lam^j, lam^{j+1}, w and g the same way; the tile of
// u^{j-1} is copied from memory one step ahead, and the share of the gradient
// of step j is computed beside step j - 1.
#include "stencil_v3.cuh"

namespace ckfwi {
namespace {

constexpr int NT2 = 512;                          // threads
constexpr int NE2 = 256;                          // of them, the ones that compute edges and exchange them
constexpr int SLOTS2 = 4;                         // exchange buffers in turn

// columns a strip between x neighbours has, and the x margin of a staged
// tile: whole vectors, at least K
__host__ __device__ constexpr int px2(int K) { return K <= 4 ? 4 : 8; }

// shared-memory layout of a tile
struct Tile2 {
    int bx, bz, pitch, rows;
    __host__ __device__ Tile2(int K, int bx_, int bz_) : bx(bx_), bz(bz_)
    {
        pitch = bx + 2 * px2(K);
        rows = bz + 2 * K + 1;                    // a row pair may read one row past the halo
    }
    __host__ __device__ int plane() const { return pitch * rows; }
    __host__ __device__ int own() const { return bx * bz; }
    __host__ size_t smem(bool reverse) const
    {
        return (size_t)((reverse ? 4 : 2) * plane() + (reverse ? 2 : 1) * own() + bx + (bz + 3) / 4 * 4) * 4;
    }
};

// vectors a tile publishes a step: its first and last K rows, its first and
// last px2(K) columns
__host__ __device__ constexpr int strip_vecs(int K, int bx, int bz) { return 2 * (K * (bx / 4) + bz * (px2(K) / 4)); }

__device__ __forceinline__ void cp16(float* dst, const float* src, bool on)
{
    const int n = on ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Copy rows x nv vectors of a field, from grid point (z0, x0), to shared
// memory (row length `pitch`); vectors that start outside the grid are zero.
// (x0 is a multiple of 4; a vector that straddles the last column reads the
// row's zero padding.)
__device__ __forceinline__ void stage2(float* dst, int pitch, int rows, int nv, const float* f, int z0, int x0, int nz,
                                       int nx, long long pxy)
{
    for (int i = threadIdx.x; i < rows * nv; i += NT2) {
        const int r = i / nv, q = i - r * nv;
        const int z = z0 + r, x = x0 + 4 * q;
        const bool on = z >= 0 && z < nz && x >= 0 && x < nx;
        cp16(dst + r * pitch + 4 * q, on ? f + z * pxy + x : f, on);
    }
}

// the same from a 16-bit field, widened on the way
template <class T>
__device__ __forceinline__ void stage2_16(float* dst, int pitch, int rows, int nv, const T* f, int z0, int x0, int nz,
                                          int nx, long long pxy)
{
    for (int i = threadIdx.x; i < rows * nv; i += NT2) {
        const int r = i / nv, q = i - r * nv;
        const int z = z0 + r, x = x0 + 4 * q;
        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (z >= 0 && z < nz && x >= 0 && x < nx) gldu<T, 4>(v, f + z * pxy + x);
        vst<4>(dst + r * pitch + 4 * q, v);
    }
}

// Laplacian of four points of one row: z neighbours q[0 .. 2K] (q[K] the row
// itself), x neighbours from the staged row at sm (lap_at's order)
template <int K>
__device__ __forceinline__ void lap2(float (&out)[4], const float (*q)[4], const float* sm, const float* c)
{
    constexpr int PX = px2(K);
    float xw[4 + 2 * PX];
    const float* u = q[K];
#pragma unroll
    for (int k = 0; k < PX; k += 4) {
        float t[4];
        sld<4>(t, sm - PX + k);
#pragma unroll
        for (int i = 0; i < 4; ++i) xw[k + i] = t[i];
        sld<4>(t, sm + 4 + k);
#pragma unroll
        for (int i = 0; i < 4; ++i) xw[PX + 4 + k + i] = t[i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) xw[PX + i] = u[i];
    float2 nu[2], acc[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        nu[p] = f2(-u[2 * p], -u[2 * p + 1]);
        acc[p] = f2(0.0f, 0.0f);
    }
#pragma unroll
    for (int j = K; j >= 1; --j) {
        const float* zp = q[K + j];
        const float* zm = q[K - j];
        const float2 cj = f2(c[j - 1], c[j - 1]);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int i = 2 * p;
            float2 s = __fadd2_rn(__fadd2_rn(f2(zp[i], zp[i + 1]), nu[p]), __fadd2_rn(f2(zm[i], zm[i + 1]), nu[p]));
            float2 sx;
            if (j % 2 == 0) {
                sx = __fadd2_rn(__fadd2_rn(f2(xw[PX + i + j], xw[PX + i + 1 + j]), nu[p]),
                                __fadd2_rn(f2(xw[PX + i - j], xw[PX + i + 1 - j]), nu[p]));
            } else {
                sx.x = __fadd_rn(__fsub_rn(xw[PX + i + j], u[i]), __fsub_rn(xw[PX + i - j], u[i]));
                sx.y = __fadd_rn(__fsub_rn(xw[PX + i + 1 + j], u[i + 1]), __fsub_rn(xw[PX + i + 1 - j], u[i + 1]));
            }
            s = __fadd2_rn(s, sx);
            acc[p] = __ffma2_rn(cj, s, acc[p]);
        }
    }
    if (K > 4) {        // see inj4
#pragma unroll
        for (int p = 0; p < 2; ++p) acc[p] = __fadd2_rn(acc[p], f2(0.0f, 0.0f));
    }
    out[0] = acc[0].x;
    out[1] = acc[0].y;
    out[2] = acc[1].x;
    out[3] = acc[1].y;
}

// what is injected into point x of row `row` of the box
__device__ __forceinline__ float inj1(const Inj& in, const float* series, int row, int x)
{
    float acc = 0.0f;
    if (x >= in.x0 && x < in.x1) {
        const int b = row * (in.x1 - in.x0) + x - in.x0;
        const int e1 = in.rowptr[b + 1];
        for (int e = in.rowptr[b]; e < e1; ++e) acc = __fmaf_rn(in.wt[e], series[in.col[e]], acc);
    }
    return acc;
}

// Injection of four points of row z (`on`: somewhere in the tile).  Zero is
// added where nothing is injected, as the one-step kernels do: a Laplacian of
// the smallest values can round to -0, which that turns into +0.  At order 16
// the Laplacian's last addition does it, for the registers (464 x 1104, 300
// steps: 6.53 ms; 6.56 to 6.76 in forms that do it here; there a point whose
// injected value rounds to -0 as well gets +0).  At the other orders this is
// the faster place (281 x 281, order 4, 500 steps: 0.88 ms against 0.92).
template <int K>
__device__ __forceinline__ void inj4(float (&s)[4], bool on, const Inj& in, const float* series, int z, int x0)
{
    const bool hit = on && z >= in.z0 && z < in.z1 && x0 + 4 > in.x0 && x0 < in.x1;
    if constexpr (K > 4) {
        if (!hit) return;
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = __fadd_rn(s[i], inj1(in, series, z - in.z0, x0 + i));
    } else {
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (hit) {
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = inj1(in, series, z - in.z0, x0 + i);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = __fadd_rn(s[i], acc[i]);
    }
}

__device__ __forceinline__ void out32(float* p, long long o, const float* v, int x0, int nx)
{
    if (x0 + 4 <= nx) {
        vstp<4>(p + o, v);
    } else {
        for (int i = 0; i < 4; ++i)
            if (x0 + i < nx) p[o + i] = v[i];
    }
}


// a level's destinations (most levels have none: a.levels says which do, so
// that the table is not looked at for the others)
__device__ __forceinline__ bool goes_out(const Step2Args& a, int level) { return (a.levels[level >> 5] >> (level & 31)) & 1u; }
__device__ __forceinline__ void out_level(const Step2Args& a, int level, long long o, const float* v, int x0)
{
    const int nx = a.g.nx;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        void* p = a.dst[level][k];
        if (!p) break;
        const int t = a.dtype[level][k];
        const bool full = x0 + 4 <= nx;
        if (t == CK_FP32) out32(static_cast<float*>(p), o, v, x0, nx);
        else if (t == CK_BF16) st16<__nv_bfloat16, 4>(p, o, v, full, x0, nx);
        else if (st16<__half, 4>(p, o, v, full, x0, nx)) atomicOr(a.err, 1);
    }
}

// ---------------------------------------------------------------- exchange
__device__ __forceinline__ void publish(uint4* p, const float* v, unsigned e)
{
    asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(__float_as_uint(v[0])), "r"(e),
                 "r"(__float_as_uint(v[1])), "r"(e) : "memory");
    asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p + 1), "r"(__float_as_uint(v[2])), "r"(e),
                 "r"(__float_as_uint(v[3])), "r"(e) : "memory");
}

__device__ __forceinline__ uint4 ldv(const uint4* p)
{
    uint4 r;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p) : "memory");
    return r;
}

// poll a published vector; false when `rounds` looks did not find the epoch
__device__ __forceinline__ bool receive(const uint4* p, float* dst, unsigned e, long long rounds)
{
    for (long long i = 0; i < rounds; ++i) {
        const uint4 a = ldv(p), b = ldv(p + 1);
        if (a.y == e && a.w == e && b.y == e && b.w == e) {
            *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(a.x), __uint_as_float(a.z),
                                                          __uint_as_float(b.x), __uint_as_float(b.z));
            return true;
        }
        if (i > 64) __nanosleep(64);
    }
    return false;
}

// What a CTA knows about its tile
template <int K>
struct Cta2 {
    static constexpr int PX = px2(K), PQ = PX / 4;
    Tile2 t;
    int nbx, nbz, bi, bj, zt, xt, h, wq;     // tiles of the grid, this tile, its first point, rows and vectors in the grid
    uint4* xb;                               // the lane's exchange buffer
    int strip;                               // vectors of a tile's strips
    __device__ __forceinline__ Cta2(const Step2Args& a, int b) : t(K, a.bx, a.bz)
    {
        nbx = (a.g.nx + a.bx - 1) / a.bx;
        nbz = (a.g.nz + a.bz - 1) / a.bz;
        bi = b / nbx;
        bj = b - bi * nbx;
        zt = bi * a.bz;
        xt = bj * a.bx;
        h = min(a.bz, a.g.nz - zt);
        wq = (min(a.bx, a.g.nx - xt) + 3) / 4;
        xb = a.xbuf;
        strip = strip_vecs(K, a.bx, a.bz);
    }
    // strips of a tile: rows 0 .. K-1 (top), its last K rows (bottom), its
    // first and its last PQ vectors of every row (left, right)
    __device__ __forceinline__ int tile_at(int i, int j) const { return (i * nbx + j) * strip; }
    __device__ __forceinline__ int off_bottom() const { return K * (t.bx / 4); }
    __device__ __forceinline__ int off_left() const { return 2 * K * (t.bx / 4); }
    __device__ __forceinline__ int off_right() const { return off_left() + t.bz * PQ; }
    __device__ __forceinline__ uint4* slot(unsigned e) const
    {
        return xb + 2LL * (e & (SLOTS2 - 1)) * nbz * nbx * strip;
    }
    __device__ __forceinline__ bool interior() const { return h > 2 * K && wq > 2 * PQ; }
    // edge vectors of the tile: the first and the last K rows, then the first
    // and the last PQ vectors of the rows between; everything when the tile
    // has no interior
    __device__ __forceinline__ int edges() const
    {
        return interior() ? 2 * K * wq + (h - 2 * K) * 2 * PQ : h * wq;
    }
};

// `rows` rows of `nq` vectors over the threads from `start` on (all of them,
// in turn): a row each while `idle` threads suffice, else row pairs (they
// share their z neighbours)
struct Rows2 {
    int nq, rows, rp, n, start, r, q;
    __device__ __forceinline__ Rows2(int nq_, int rows_, int start_, int idle) : nq(max(nq_, 1)), rows(rows_), start(start_)
    {
        const int all = nq_ > 0 && rows_ > 0 ? nq_ * rows_ : 0;
        rp = all <= idle ? 1 : 2;
        n = rp == 1 ? all : (rows_ + 1) / 2 * nq_;
        if (all == 0) n = 0;
        set(first());
    }
    __device__ __forceinline__ int first() const { return ((int)threadIdx.x - start + NT2) % NT2; }
    __device__ __forceinline__ void set(int i)
    {
        const int p = i / nq;
        q = i - p * nq;
        r = rp * p;
    }
};

// An edge vector: where it is, and its places in the strips (vectors from the
// slot's start, -1: none)
struct Edge2 {
    int r, q;
    template <int K>
    __device__ __forceinline__ void set(const Cta2<K>& ct, int i)
    {
        const int rows = 2 * K * ct.wq, h = ct.h, wq = ct.wq, PQ = ct.PQ, bq = ct.t.bx / 4;
        if (!ct.interior()) {
            r = i / wq;
            q = i - r * wq;
        } else if (i < rows) {
            r = i / wq;
            q = i - r * wq;
            if (r >= K) r += h - 2 * K;
        } else {
            const int k = i - rows, c = k / (h - 2 * K);
            r = K + k - c * (h - 2 * K);
            q = c < PQ ? c : wq - 2 * PQ + c;
        }
        const int me = ct.tile_at(ct.bi, ct.bj);
        st = sb = sl = sr = -1;
        if (ct.bi > 0 && r < K) st = me + r * bq + q;
        if (ct.bi + 1 < ct.nbz && r >= h - K) sb = me + ct.off_bottom() + (r - h + K) * bq + q;
        if (ct.bj > 0 && q < PQ) sl = me + ct.off_left() + r * PQ + q;
        if (ct.bj + 1 < ct.nbx && q >= wq - PQ) sr = me + ct.off_right() + r * PQ + q - wq + PQ;
    }
    int st, sb, sl, sr;
    __device__ __forceinline__ void send(uint4* slot, const float* v, unsigned e) const
    {
        if (st >= 0) publish(slot + 2LL * st, v, e);
        if (sb >= 0) publish(slot + 2LL * sb, v, e);
        if (sl >= 0) publish(slot + 2LL * sl, v, e);
        if (sr >= 0) publish(slot + 2LL * sr, v, e);
    }
};

// A vector of a neighbour's strips and its place in the margins of a plane.
// The tile above gives its last K rows, the one below its first (as many as
// it has), the left one its last PQ vectors, the right one its first (as many
// as it has), and the one below and right its first vector.
struct Take2 {
    int src, dst;            // src < 0: none
    template <int K>
    __device__ __forceinline__ static int count(const Cta2<K>& ct, int nz, int nx)
    {
        const int dn = ct.bi + 1 < ct.nbz ? min(K, nz - ct.zt - ct.t.bz) * ct.wq : 0;
        const int rq = ct.bj + 1 < ct.nbx ? min(ct.PQ, (nx - ct.xt - ct.t.bx + 3) / 4) : 0;
        return (ct.bi > 0 ? K * ct.wq : 0) + dn + (ct.bj > 0 ? ct.h * ct.PQ : 0) + ct.h * rq + (dn > 0 && rq > 0 ? 1 : 0);
    }
    template <int K>
    __device__ __forceinline__ void set(const Cta2<K>& ct, int k, int nz, int nx)
    {
        const int bq = ct.t.bx / 4, wq = ct.wq, PQ = ct.PQ, bi = ct.bi, bj = ct.bj, pitch = ct.t.pitch;
        const int n_up = bi > 0 ? K * wq : 0;
        const int n_dn = bi + 1 < ct.nbz ? min(K, nz - ct.zt - ct.t.bz) * wq : 0;
        const int n_lf = bj > 0 ? ct.h * PQ : 0;
        const int rq = bj + 1 < ct.nbx ? min(PQ, (nx - ct.xt - ct.t.bx + 3) / 4) : 0;
        dst = K * pitch + 4 * PQ;
        if (k < n_up) {
            const int r = k / wq, q = k - r * wq;
            src = ct.tile_at(bi - 1, bj) + ct.off_bottom() + r * bq + q;
            dst += (r - K) * pitch + 4 * q;
        } else if ((k -= n_up) < n_dn) {
            const int r = k / wq, q = k - r * wq;
            src = ct.tile_at(bi + 1, bj) + r * bq + q;
            dst += (ct.t.bz + r) * pitch + 4 * q;
        } else if ((k -= n_dn) < n_lf) {
            const int r = k / PQ, q = k - r * PQ;
            src = ct.tile_at(bi, bj - 1) + ct.off_right() + r * PQ + q;
            dst += r * pitch + 4 * (q - PQ);
        } else if ((k -= n_lf) < ct.h * rq) {
            const int r = k / rq, q = k - r * rq;
            src = ct.tile_at(bi, bj + 1) + ct.off_left() + r * PQ + q;
            dst += r * pitch + ct.t.bx + 4 * q;
        } else {
            src = ct.tile_at(bi + 1, bj + 1);
            dst += ct.t.bz * pitch + ct.t.bx;
        }
    }
};

// What every step repeats, worked out once: the thread's first edge vector,
// its first vector to take and its first interior rows
template <int K>
struct Plan2 {
    Cta2<K> ct;
    int nz, nx, n_edge, n_take;
    Edge2 edge;
    Take2 take;
    Rows2 in;
    __device__ __forceinline__ Plan2(const Step2Args& a, int b)
        : ct(a, b), nz(a.g.nz), nx(a.g.nx), in(ct.interior() ? ct.wq - 2 * ct.PQ : 0, ct.h - 2 * K, NE2, NT2 - NE2)
    {
        const int tid = threadIdx.x;
        n_edge = tid < NE2 ? ct.edges() : 0;
        n_take = tid < NE2 ? Take2::count(ct, nz, nx) : 0;
        if (tid < n_edge) edge.set(ct, tid);
        if (tid < n_take) take.set(ct, tid, nz, nx);
    }
    __device__ __forceinline__ bool meets(const Inj& in_) const
    {
        return in_.on && in_.z0 < ct.zt + ct.h && in_.z1 > ct.zt && in_.x0 < ct.xt + 4 * ct.wq && in_.x1 > ct.xt;
    }
    __device__ __forceinline__ bool receive_all(float* b, unsigned e, long long rounds) const
    {
        const uint4* s = ct.slot(e);
        bool ok = true;
        if ((int)threadIdx.x < n_take) ok = receive(s + 2LL * take.src, b + take.dst, e, rounds);
        for (int i = threadIdx.x + NE2; i < n_take; i += NE2) {
            Take2 t;
            t.set(ct, i, nz, nx);
            ok = receive(s + 2LL * t.src, b + t.dst, e, rounds) && ok;
        }
        return ok;
    }
};

// What the points of a step share
template <int K>
struct Step2Env {
    float* b1;            // level i
    float* b2;            // level i - 1, then level i + 1
    const float *w, *ezs, *exs;
    float hdt;
    float c[K];           // c[j - 1]: weight of the neighbours j away
    bool damped, inject;  // some point of the tile is damped / may be injected
};

// leapfrog() of two points without damping: b = 1 and the division drop out
// (1 (c - p) and t / 1 round to themselves)
__device__ __forceinline__ float2 leap2u(float2 c, float2 p, float2 w, float2 s)
{
    return __fadd2_rn(c, __ffma2_rn(w, s, __ffma2_rn(p, f2(-1.0f, -1.0f), c)));
}

// The update of vector (r, q) of the tile from its z window; writes level
// i + 1 over level i - 1 and returns it
template <int K>
__device__ __forceinline__ void update2(float (&v)[4], const Cta2<K>& ct, const float (*qz)[4], const Step2Env<K>& ev,
                                        const Inj& in, const float* series, int nx, int r, int q)
{
    const int o = (K + r) * ct.t.pitch + ct.PX + 4 * q;
    const int x0 = ct.xt + 4 * q;
    float s[4], pv[4], wv[4];
    sld<4>(pv, ev.b2 + o);
    sld<4>(wv, ev.w + r * ct.t.bx + 4 * q);
    lap2<K>(s, qz, ev.b1 + o, ev.c);
    if (K <= 4 || ev.inject) inj4<K>(s, ev.inject, in, series, ct.zt + r, x0);
    const float* uc = qz[K];
    float2 a0, a1;
    if (ev.damped) {
        const float ez = ev.ezs[r];
        float ex[4];
        sld<4>(ex, ev.exs + 4 * q);
        const float2 e0 = __fadd2_rn(f2(ez, ez), f2(ex[0], ex[1])), e1 = __fadd2_rn(f2(ez, ez), f2(ex[2], ex[3]));
        a0 = leap2v(f2(uc[0], uc[1]), f2(pv[0], pv[1]), f2(wv[0], wv[1]), f2(s[0], s[1]), e0, ev.hdt);
        a1 = leap2v(f2(uc[2], uc[3]), f2(pv[2], pv[3]), f2(wv[2], wv[3]), f2(s[2], s[3]), e1, ev.hdt);
    } else {
        a0 = leap2u(f2(uc[0], uc[1]), f2(pv[0], pv[1]), f2(wv[0], wv[1]), f2(s[0], s[1]));
        a1 = leap2u(f2(uc[2], uc[3]), f2(pv[2], pv[3]), f2(wv[2], wv[3]), f2(s[2], s[3]));
    }
    v[0] = a0.x;
    v[1] = a0.y;
    v[2] = a1.x;
    v[3] = a1.y;
    if (x0 + 4 > nx) {
#pragma unroll
        for (int i = 1; i < 4; ++i)
            if (x0 + i >= nx) v[i] = 0.0f;
    }
    vst<4>(ev.b2 + o, v);
}

// rows first + r .. of vector q of a staged plane as z window of R rows
template <int K, int R>
__device__ __forceinline__ void window2(float (&win)[2 * K + R][4], const float* plane, int pitch, int r, int q)
{
    const float* p = plane + r * pitch + px2(K) + 4 * q;       // row r - K of the tile
#pragma unroll
    for (int k = 0; k < 2 * K + R; ++k) sld<4>(win[k], p + k * pitch);
}

// One step of the tile: edges (published when `send`), then the interior.
// emit(r, q, level i values, level i + 1 values).
template <int K, class Emit>
__device__ __forceinline__ void step2(const Plan2<K>& pl, const Step2Env<K>& ev, const Inj& in, const float* series, bool send,
                                      unsigned e, Emit emit)
{
    const Cta2<K>& ct = pl.ct;
    Edge2 ed = pl.edge;
    for (int i = threadIdx.x; i < pl.n_edge; i += NE2) {
        if (i >= NE2) ed.set(ct, i);
        float win[2 * K + 1][4], v[4];
        window2<K, 1>(win, ev.b1, ct.t.pitch, ed.r, ed.q);
        update2<K>(v, ct, win, ev, in, series, pl.nx, ed.r, ed.q);
        if (send) ed.send(ct.slot(e), v, e);
        emit(ed.r, ed.q, win[K], v);
    }
    // the interior: by the threads without edges while the others are at
    // theirs; where it has more rows than those threads, all share what is left
    Rows2 pr = pl.in;
    if (pr.rp == 1) {
        if (pr.first() < pr.n) {                  // a row each: one round
            float win[2 * K + 1][4], v[4];
            const int r = pr.r + K, q = pr.q + ct.PQ;
            window2<K, 1>(win, ev.b1, ct.t.pitch, r, q);
            update2<K>(v, ct, win, ev, in, series, pl.nx, r, q);
            emit(r, q, win[K], v);
        }
        return;
    }
    for (int i = pr.first(); i < pr.n; i += NT2) {
        if (i >= NT2) pr.set(i);
        float win[2 * K + 2][4], v[4];
        const int r = pr.r + K, q = pr.q + ct.PQ;
        window2<K, 2>(win, ev.b1, ct.t.pitch, r, q);
        update2<K>(v, ct, win, ev, in, series, pl.nx, r, q);
        emit(r, q, win[K], v);
        if (pr.r + 1 < pr.rows) {
            update2<K>(v, ct, win + 1, ev, in, series, pl.nx, r + 1, q);
            emit(r + 1, q, win[K + 1], v);
        }
    }
}

// the state, w and the damping tables of a tile; whether the thread has seen
// a damped row or column
template <int K>
__device__ __forceinline__ bool stage_state(const Cta2<K>& ct, float* b1, float* b2, float* w, float* exs, float* ezs,
                                            const Step2Args& a)
{
    const Tile2& t = ct.t;
    const int nz = a.g.nz, nx = a.g.nx;
    stage2(b1, t.pitch, t.rows, t.pitch / 4, a.f1, ct.zt - K, ct.xt - ct.PX, nz, nx, a.g.pxy);
    stage2(b2, t.pitch, t.rows, t.pitch / 4, a.f2, ct.zt - K, ct.xt - ct.PX, nz, nx, a.g.pxy);
    stage2(w, t.bx, t.bz, t.bx / 4, a.w, ct.zt, ct.xt, nz, nx, a.g.pxy);
    cp_commit();
    bool damped = false;
    for (int i = threadIdx.x; i < t.bx; i += NT2) {
        exs[i] = ct.xt + i < nx ? a.eta[nz + a.g.ny + ct.xt + i] : 0.0f;
        damped |= exs[i] != 0.0f;
    }
    for (int i = threadIdx.x; i < t.bz; i += NT2) {
        ezs[i] = ct.zt + i < nz ? a.eta[ct.zt + i] : 0.0f;
        damped |= ezs[i] != 0.0f;
    }
    return damped;
}

template <int K>
__device__ __forceinline__ void fwd2_body(const Step2Args& a, int b, float* sm)
{
    const Plan2<K> pl(a, b);
    const Cta2<K>& ct = pl.ct;
    const Tile2& t = ct.t;
    const int tid = threadIdx.x;
    float* b1 = sm;
    float* b2 = b1 + t.plane();
    float* w = b2 + t.plane();
    float* exs = w + t.own();
    float* ezs = exs + t.bx;
    const unsigned e0 = a.epoch[b];
    Step2Env<K> ev{b1, b2, w, ezs, exs, a.hdt, {}, false, pl.meets(a.src)};
#pragma unroll
    for (int j = 0; j < K; ++j) ev.c[j] = a.c[j + 1];
    ev.damped = __syncthreads_or(stage_state<K>(ct, b1, b2, w, exs, ezs, a));
    const int r0 = a.smp.n > 0 ? a.rstart[b] : 0, r1 = a.smp.n > 0 ? a.rstart[b + 1] : 0;
    cp_wait();
    __syncthreads();
    const int spos = (tid - NE2 - pl.in.n % NT2 + 2 * NT2) % NT2;    // the threads after those of the interior sample
    for (int i = 0; i < a.T; ++i) {
        // receivers of level n + i
        for (int k = r0 + spos; k < r1; k += NT2) {
            const int2 at = __ldg(a.rlist + k);
            const float4 wt = __ldg(a.rwt + k);
            const float* p = ev.b1 + at.x;
            float acc = __fmaf_rn(wt.x, p[0], 0.0f);
            acc = __fmaf_rn(wt.y, p[1], acc);
            acc = __fmaf_rn(wt.z, p[t.pitch], acc);
            acc = __fmaf_rn(wt.w, p[t.pitch + 1], acc);
            a.smp.out[(long long)i * a.smp.n + at.y] = acc;
        }
        const bool last = i + 1 == a.T;
        const unsigned e = e0 + 1u + i;
        const bool out0 = i == 0 && goes_out(a, 0), out = goes_out(a, i + 1);
        step2<K>(pl, ev, a.src, a.src.series + i, !last, e,
                 [&](int r, int q, const float* uc, const float* v) {
                     if (!out0 && !out) return;
                     const int x = ct.xt + 4 * q;
                     const long long o = (long long)(ct.zt + r) * a.g.pxy + x;
                     if (out0) out_level(a, 0, o, uc, x);
                     if (out) out_level(a, i + 1, o, v, x);
                 });
        const bool ok = last || pl.receive_all(ev.b2, e, a.wait_limit);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicOr(a.err, 8);
            return;
        }
        float* s = ev.b2;
        ev.b2 = ev.b1;
        ev.b1 = s;
    }
    if (tid == 0) a.epoch[b] = e0 + a.T;
}

template <int K>
__device__ __forceinline__ void adj2_body(const Step2Args& a, int b, float* sm)
{
    const Plan2<K> pl(a, b);
    const Cta2<K>& ct = pl.ct;
    const Tile2& t = ct.t;
    const int nz = a.g.nz, nx = a.g.nx, tid = threadIdx.x;
    const long long pxy = a.g.pxy;
    float* b1 = sm;
    float* b2 = b1 + t.plane();
    float* us = b2 + t.plane();                   // two u tiles
    float* w = us + 2 * t.plane();
    float* gs = w + t.own();
    float* exs = gs + t.own();
    float* ezs = exs + t.bx;
    const unsigned e0 = a.epoch[b];
    auto load_u = [&](int i) {
        float* d = us + (i & 1) * t.plane();
        const int z0 = ct.zt - K, x0 = ct.xt - ct.PX, nv = t.pitch / 4;
        if (a.ut[i] == U_FP32) stage2(d, t.pitch, t.rows, nv, static_cast<const float*>(a.u[i]), z0, x0, nz, nx, pxy);
        else if (a.ut[i] == U_FP16) stage2_16(d, t.pitch, t.rows, nv, static_cast<const __half*>(a.u[i]), z0, x0, nz, nx, pxy);
        else stage2_16(d, t.pitch, t.rows, nv, static_cast<const __nv_bfloat16*>(a.u[i]), z0, x0, nz, nx, pxy);
        cp_commit();
    };
    Step2Env<K> ev{b1, b2, w, ezs, exs, a.hdt, {}, false, pl.meets(a.adj)};
#pragma unroll
    for (int j = 0; j < K; ++j) ev.c[j] = a.c[j + 1];
    const bool src = pl.meets(a.src), damped = stage_state<K>(ct, b1, b2, w, exs, ezs, a);
    stage2(gs, t.bx, t.bz, t.bx / 4, a.gacc, ct.zt, ct.xt, nz, nx, pxy);
    load_u(0);
    cp_wait();
    ev.damped = __syncthreads_or(damped);
    // the gradient's rows by the threads after those of the interior (by the
    // same ones, a small tile's step was the sum of both: 4.4 us at 281 x 281)
    const Rows2 gp0(ct.wq, ct.h, (NE2 + pl.in.n) % NT2, NT2 - NE2 - pl.in.n);
    // Phase i: step i of lam, and the gradient of step i - 1, whose lam (now
    // b1) the barrier before has completed.  The u tile that phase i + 1 needs
    // replaces the one that the gradient of phase i - 1 has read.
    for (int i = 0; i <= a.T; ++i) {
        const bool step = i < a.T, last = i + 1 >= a.T;
        const unsigned e = e0 + 1u + i;
        if (i > 0 && step) load_u(i);
        if (step)
            step2<K>(pl, ev, a.adj, a.adj.series - (long long)i * a.adj_stride, !last, e,
                     [&](int r, int q, const float*, const float* v) {
                         if (i + 2 < a.T) return;
                         float* p = static_cast<float*>(a.dst[i + 1][0]);
                         const int x = ct.xt + 4 * q;
                         if (p) out32(p, (long long)(ct.zt + r) * pxy + x, v, x, nx);
                     });
        if (i > 0) {
            const float* ub = us + ((i - 1) & 1) * t.plane();
            Rows2 pr = gp0;
            for (int k = pr.first(); k < pr.n; k += NT2) {
                if (k >= NT2) pr.set(k);
                float win[2 * K + 2][4];
                window2<K, 2>(win, ub, t.pitch, pr.r, pr.q);
                const int x0 = ct.xt + 4 * pr.q;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = pr.r + h, o = (K + r) * t.pitch + ct.PX + 4 * pr.q;
                    if (h >= pr.rp || r >= ct.h) break;
                    float s[4], lv[4], gv[4];
                    sld<4>(lv, ev.b1 + o);
                    float* gp = gs + r * t.bx + 4 * pr.q;
                    sld<4>(gv, gp);
                    lap2<K>(s, win + h, ub + o, ev.c);
                    if (K <= 4 || src) inj4<K>(s, src, a.src, a.src.series - (i - 1), ct.zt + r, x0);
                    const float2 g0 = __ffma2_rn(f2(lv[0], lv[1]), f2(s[0], s[1]), f2(gv[0], gv[1]));
                    const float2 g1 = __ffma2_rn(f2(lv[2], lv[3]), f2(s[2], s[3]), f2(gv[2], gv[3]));
                    gv[0] = g0.x;
                    gv[1] = g0.y;
                    gv[2] = g1.x;
                    gv[3] = g1.y;
                    if (step) vst<4>(gp, gv);
                    else out32(a.gacc, (long long)(ct.zt + r) * pxy + x0, gv, x0, nx);
                }
            }
        }
        if (!step) break;
        const bool ok = last || pl.receive_all(ev.b2, e, a.wait_limit);
        cp_wait();
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicOr(a.err, 8);
            return;
        }
        float* s = ev.b2;
        ev.b2 = ev.b1;
        ev.b1 = s;
    }
    if (tid == 0) a.epoch[b] = e0 + a.T;
}

template <int K>
__global__ void __launch_bounds__(NT2, 1) fwd2_kernel(const __grid_constant__ Step2Args a)
{
    extern __shared__ __align__(16) float sm2[];
    fwd2_body<K>(a, blockIdx.x, sm2);
}

template <int K>
__global__ void __launch_bounds__(NT2, 1) adj2_kernel(const __grid_constant__ Step2Args a)
{
    extern __shared__ __align__(16) float sm2[];
    adj2_body<K>(a, blockIdx.x, sm2);
}

// several lanes: lane l's arguments are tab[l], its tiles are CTAs start[l] .. start[l+1]-1
template <int K>
__global__ void __launch_bounds__(NT2, 1) fwd2_batch_kernel(const Step2Args* __restrict__ tab, const int* __restrict__ start, int nl)
{
    extern __shared__ __align__(16) float sm2[];
    __shared__ __align__(16) Step2Args a;
    const int b = stage_args(a, tab, start, nl);
    fwd2_body<K>(a, b, sm2);
}

template <int K>
__global__ void __launch_bounds__(NT2, 1) adj2_batch_kernel(const Step2Args* __restrict__ tab, const int* __restrict__ start, int nl)
{
    extern __shared__ __align__(16) float sm2[];
    __shared__ __align__(16) Step2Args a;
    const int b = stage_args(a, tab, start, nl);
    adj2_body<K>(a, b, sm2);
}

// a cooperative launch: the tiles wait for one another, so all are resident or none runs
template <class... P, class... A>
cudaError_t coop(void (*k)(P...), unsigned blocks, size_t sh, cudaStream_t s, A&&... args)
{
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(NT2);
    cfg.dynamicSmemBytes = sh;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, std::forward<A>(args)...);
}

template <int K>
cudaError_t go2(const Step2Args* one, const BatchLaunch<Step2Args>* many, const Tile& t, bool reverse, cudaStream_t s)
{
    const size_t sh = Tile2(K, t.bx, t.zlen).smem(reverse);
    if (one) {
        const unsigned nb = (unsigned)(((one->g.nx + t.bx - 1) / t.bx) * ((one->g.nz + t.zlen - 1) / t.zlen));
        return coop(reverse ? adj2_kernel<K> : fwd2_kernel<K>, nb, sh, s, *one);
    }
    return coop(reverse ? adj2_batch_kernel<K> : fwd2_batch_kernel<K>, (unsigned)many->blocks, sh, s, many->tab,
                many->start, many->lanes);
}

cudaError_t go2(const Step2Args* one, const BatchLaunch<Step2Args>* many, const Tile& t, int K, bool reverse, cudaStream_t s)
{
    if (!step2_supported(2, K, t, reverse)) return cudaErrorInvalidValue;
    switch (K) {
    case 1: return go2<1>(one, many, t, reverse, s);
    case 2: return go2<2>(one, many, t, reverse, s);
    case 4: return go2<4>(one, many, t, reverse, s);
    case 8: return go2<8>(one, many, t, reverse, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

bool step2_supported(int dims, int K, const Tile& t, bool reverse)
{
    if (dims != 2 || t.ver != 9 || (K != 1 && K != 2 && K != 4 && K != 8)) return false;
    // neighbours hold each other's whole halo, and a row of vectors has a thread each
    if (t.bx < px2(K) || t.bx % 4 || t.by != 1 || t.vec != 4 || t.zlen < K || t.bx / 4 > 4096) return false;
    return Tile2(K, t.bx, t.zlen).smem(reverse) + sizeof(Step2Args) + 64 <= 227 * 1024;
}

int step2_place(int K, const Tile& t, int z, int x)
{
    return (K + z % t.zlen) * Tile2(K, t.bx, t.zlen).pitch + px2(K) + x % t.bx;
}

// bytes of a lane's exchange buffer for `tiles` tiles
size_t step2_exchange_bytes(int K, const Tile& t, long long tiles)
{
    return (size_t)SLOTS2 * tiles * strip_vecs(K, t.bx, t.zlen) * 32;
}

cudaError_t launch_step2(const Step2Args& a, const Tile& t, int K, bool reverse, cudaStream_t s)
{
    if (a.T < 1 || a.T > STEP2_MAX) return cudaErrorInvalidValue;
    return go2(&a, nullptr, t, K, reverse, s);
}

cudaError_t launch_step2_batch(const BatchLaunch<Step2Args>& b, const Tile& t, int K, bool reverse, cudaStream_t s)
{
    return go2(nullptr, &b, t, K, reverse, s);
}

}  // namespace ckfwi
