// Fixed-rate mode of the block codec (Sec. 2.2 lists ZFP's fixed-rate mode
// beside the fixed-tolerance one: a guaranteed size, no error bound).
//
//  rate     R bits per value, 1 <= R <= 32; every block occupies exactly
//           W = ceil(R 4^d / 32) words, a budget of 32 W bits, so a field
//           takes 16 + nblocks W words whatever its values.
//  block    0: all values +-0, a non-finite value (flag NONFINITE) or
//           Emax < -100 (values below 2^-99 are flushed); rest of the
//           budget zero.  Else 1, Emax+127 (8), ptop (5), then planes ptop
//           down to 0 coded as in the fixed-accuracy mode (verbatim bits of
//           the s significant coefficients, then group tests) until the
//           budget is full: the first bit that does not fit is dropped and
//           coding stops.  Integers, lifting, order and negabinary are the
//           fixed-accuracy mode's (codec_common.cuh).
//  decode   the same bits up to the budget; bits not read are zero;
//           x_hat = float(i_hat) 2^(Emax-23).
//  container header words of the fixed-accuracy mode with version 2,
//           [7] = nblocks W, [8] = R; the blocks back to back after it.
//
// GPU layout: one thread per block, as in the fixed-accuracy kernels.  The
// block's values live in registers (lifting, order and negabinary with
// compile-time indices); two 32 x 32 bit transposes turn the 64 coefficient
// words into 32 plane masks of 64 bits, kept in shared memory so that the
// coder can walk the planes with a run-time index.  On a 64-bit plane mask
// the verbatim bits are one masked append and a group test plus its run is
// one find-first-set.  The decoder parses the planes into the same masks
// and transposes them back.  No size table and no scan: block b sits at
// word 16 + b W of the stream.
#include "codec_common.cuh"

namespace ckfwi {
namespace {

constexpr uint32_t RATE_VERSION = VERSION_RATE;
constexpr int RATE_EMIN = -100;
constexpr int RT = 64;                 // threads (blocks) per CTA

__host__ __device__ inline long long rate_block_words(int dims, int rate) { return ((long long)rate * (dims == 3 ? 64 : 16) + 31) / 32; }

// Bit writer straight into the block's words: the low n bits of v (n <= 32,
// nothing above them).  The caller keeps the budget.
struct RateW {
    uint32_t* o;
    unsigned long long acc;
    int nacc;
    __device__ __forceinline__ void put(uint32_t v, int n)
    {
        acc |= (unsigned long long)v << nacc;
        nacc += n;
        if (nacc >= 32) {
            *o++ = (uint32_t)acc;
            acc >>= 32;
            nacc -= 32;
        }
    }
    __device__ __forceinline__ void put64(unsigned long long v, int n)   // n <= 64, bits above n ignored
    {
        if (n > 32) {
            put((uint32_t)v, 32);
            put((uint32_t)(v >> 32) & mask32(n - 32), n - 32);
        } else if (n > 0) {
            put((uint32_t)v & mask32(n), n);
        }
    }
    __device__ __forceinline__ void finish(uint32_t* end)   // the partial word, then zeros to the budget
    {
        if (nacc > 0) *o++ = (uint32_t)acc;
        while (o < end) *o++ = 0u;
    }
};

// First word of field `fld`'s stream: a lane's second stream follows its
// first (every stream has the same length), which starts at the word in
// base[from[0]]; a stream that does not fit the pool takes no room.
__device__ __forceinline__ long long rate_base(const CodecCall& c, const CodecLane& A, int fld, long long total)
{
    const long long b = A.base[c.from[0]];
    return fld && b + total <= A.cap_words ? b + total : b;
}

// The 16 header words, the pool's next word and the statistics of every
// field of a call, before its blocks are coded (a block with a non-finite
// value marks the header).
__global__ void rate_header_kernel(const __grid_constant__ CodecCall c)
{
    int fld;
    const CodecLane& A = item_of(c, fld);
    const Geo G = geo_of(A.v);
    const long long total = HDR + G.nblocks * rate_block_words(G.dims, c.rate);
    const long long base = rate_base(c, A, fld, total);
    const bool fits = base + total <= A.cap_words;
    if (threadIdx.x == 0) {
        if (!fits) atomicOr(A.err, 2);
        if (fld + 1 < c.nf) A.base[c.from[1]] = fits ? base + total : base;
        else end_streams(c, A, fits ? base + total : base);
        if (fits && A.stat) A.stat[c.stat0 + fld] = (unsigned long long)total;
    }
    if (fits && threadIdx.x < HDR) {
        uint32_t h = 0;
        switch (threadIdx.x) {
        case 0: h = MAGIC; break;
        case 1: h = (uint32_t)G.dims | (RATE_VERSION << 8); break;
        case 2: h = (uint32_t)G.nz; break;
        case 3: h = (uint32_t)G.ny; break;
        case 4: h = (uint32_t)G.nx; break;
        case 5: h = (uint32_t)G.nblocks; break;
        case 7: h = (uint32_t)(total - HDR); break;
        case 8: h = (uint32_t)c.rate; break;
        default: h = 0;
        }
        A.pool[base + threadIdx.x] = h;
    }
}

// (Eight CTAs an SM, 128 registers: 59 us for a field of 187 x 213 x 229 at 16
// bits a value, 70 us with the 147 registers of no bound; 82 us with a writer
// that looped over every append, and 89 us for the decoder that looked at the
// stream anew for every group test, now 66.)
template <int DIMS>
__global__ void __launch_bounds__(RT, 8) rate_enc_kernel(const __grid_constant__ CodecCall call)
{
    constexpr int V = Cfg<DIMS>::V;
    constexpr Perm P = make_perm(DIMS);
    __shared__ unsigned long long spl[32][RT];      // plane masks of each thread's block
    int fld;
    const CodecLane& A = item_of(call, fld);
    const Geo G = geo_of(A.v);
    const int tid = threadIdx.x;
    const long long b = (long long)blockIdx.x * RT + tid;
    if (b >= G.nblocks) return;
    const int W = (int)rate_block_words(DIMS, call.rate);
    const long long total = HDR + G.nblocks * W;
    const long long base = rate_base(call, A, fld, total);
    if (base + total > A.cap_words) return;                 // the header kernel raised the error
    uint32_t* o = A.pool + base + HDR + b * W;

    float f[V];
    gather<DIMS>(A.f[call.src[fld]], A.v, block_pos(G, b), f);
    bool bad = false;
    int emax = -1000;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const uint32_t u = __float_as_uint(f[i]);
        bad = bad || !isfinite(f[i]);
        const int be = (int)((u >> 23) & 0xFF);
        if ((u & 0x7FFFFFFFu) != 0) emax = max(emax, (be > 0 ? be : 1) - 127);
    }
    if (bad || emax < RATE_EMIN) {           // zero-coded block (no non-zero value: emax = -1000)
        if (bad) {
            atomicOr(A.err, 1);
            atomicOr(A.pool + base + 9, 1u);
        }
        for (int k = 0; k < W; ++k) o[k] = 0u;
        return;
    }
    int32_t iv[V];
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const uint32_t u = __float_as_uint(f[i]);
        const int be = (int)((u >> 23) & 0xFF);
        const uint32_t M = (u & 0x7FFFFFu) | (be > 0 ? 0x800000u : 0u);
        const int sh = emax - ((be > 0 ? be : 1) - 127);
        uint32_t mag = sh >= 32 ? 0u : (M >> sh);
        if ((u & 0x7FFFFFFFu) == 0) mag = 0;
        iv[i] = (u >> 31) ? -(int32_t)mag : (int32_t)mag;
    }
    xform_fwd<DIMS>(iv);
    uint32_t lo[32], hi[32], orall = 0;
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        lo[r] = r < V ? nega(iv[P.p[r]]) : 0u;
        hi[r] = r + 32 < V ? nega(iv[P.p[r + 32 < V ? r + 32 : 0]]) : 0u;
        orall |= lo[r] | hi[r];
    }
    const int ptop = orall ? 31 - __clz(orall) : 0;
    transpose32(lo);
    if (V > 32) transpose32(hi);
#pragma unroll
    for (int p = 0; p < 32; ++p) spl[p][tid] = (unsigned long long)lo[p] | ((unsigned long long)hi[p] << 32);

    // Every append is a masked shift into the accumulator and at most one
    // store; the budget is one comparison an append, its end one partial
    // append (the first bit that does not fit is dropped and coding stops).
    RateW wr{o, 0ull, 0};
    wr.put(1u | (uint32_t)(emax + 127) << 1 | (uint32_t)ptop << 9, 14);    // fits the smallest budget, 32 bits
    int left = 32 * W - 14;
    int sgn = 0;   // coefficients already significant
#pragma unroll 1
    for (int p = ptop; p >= 0; --p) {
        const unsigned long long m = spl[p][tid];
        if (sgn > left) {
            wr.put64(m, left);
            break;
        }
        wr.put64(m, sgn);
        left -= sgn;
        bool full = false;
        while (sgn < V) {
            const unsigned long long rest = m >> sgn;
            if (!rest) {
                full = left < 1;
                if (!full) {
                    wr.put(0u, 1);
                    --left;
                }
                break;
            }
            // a group test (1), the zeros before the next significant one, and it
            const int fz = __ffsll((long long)rest) - 1;
            if (fz + 2 > left) {
                if (left > 0) {
                    wr.put(1u, 1);
                    wr.put64(0ull, left - 1);
                }
                full = true;
                break;
            }
            if (fz <= 30) {
                wr.put(1u | 2u << fz, fz + 2);
            } else {
                wr.put(1u, 1);
                wr.put64(1ull << fz, fz + 1);
            }
            left -= fz + 2;
            sgn += fz + 1;
        }
        if (full) break;
    }
    wr.finish(o + W);
}

template <int DIMS>
__global__ void __launch_bounds__(RT) rate_dec_kernel(const __grid_constant__ CodecCall call)
{
    constexpr int V = Cfg<DIMS>::V;
    constexpr Perm P = make_perm(DIMS);
    __shared__ unsigned long long spl[32][RT];
    int fld;
    const CodecLane& A = item_of(call, fld);
    const CodecView& v = A.v;
    const Geo G = geo_of(v);
    const uint32_t* __restrict__ in = A.pool;
    float* __restrict__ x = A.f[call.src[fld]];
    int* err = A.err;
    const long long cap_words = A.cap_words;
    const int tid = threadIdx.x;
    const long long b = (long long)blockIdx.x * RT + tid;
    if (b >= G.nblocks) return;
    const long long base = A.base[call.from[fld]];
    int rate = call.rate;
    if (call.any) {                                  // a whole stream from the first word on: the header is there
        if ((__ldg(in + base + 1) >> 8) != RATE_VERSION) return;
        const uint32_t r = __ldg(in + base + 8);
        if (r < 1u || r > 32u) {
            atomicOr(err, 4);
            return;
        }
        rate = (int)r;
    }
    const int W = (int)rate_block_words(DIMS, rate);
    if (base < 0 || base + HDR + G.nblocks * W > cap_words) {
        atomicOr(err, 4);
        return;
    }
    const uint32_t* h = in + base;
    if (__ldg(h) != MAGIC || __ldg(h + 1) != ((uint32_t)DIMS | (RATE_VERSION << 8)) || __ldg(h + 2) != (uint32_t)G.nz ||
        __ldg(h + 3) != (uint32_t)G.ny || __ldg(h + 4) != (uint32_t)G.nx || __ldg(h + 5) != (uint32_t)G.nblocks ||
        __ldg(h + 7) != (uint32_t)(G.nblocks * W) || __ldg(h + 8) != (uint32_t)rate) {
        atomicOr(err, 4);
        return;
    }
    const uint32_t* words = h + HDR + b * W;
    BitR rd(words, words + W, 0);
    int left = 32 * W;                             // bits of the budget not read yet
    float f[V];
    const bool coded = rd.take(1) != 0;
    if (!coded) {
#pragma unroll
        for (int i = 0; i < V; ++i) f[i] = 0.0f;
    } else {
        const int emax = (int)rd.take(8) - 127;
        const int ptop = (int)rd.take(5);
        left -= 14;
#pragma unroll
        for (int p = 0; p < 32; ++p) spl[p][tid] = 0ull;
        int sgn = 0;
        bool more = true;
#pragma unroll 1
        for (int p = ptop; p >= 0 && more; --p) {
            // verbatim bits of the significant coefficients (as many as the budget holds)
            const int k = min(sgn, left);
            unsigned long long m = k > 0 ? rd.take64(k) : 0ull;
            left -= k;
            more = k == sgn;
            while (more && sgn < V) {
                more = left > 0;
                if (!more) break;
                --left;
                if (!rd.take(1)) break;
                // coefficients sgn, sgn+1, ... up to and including the first set one
                const int avail = min(V - sgn, left);
                const int z = rd.run(avail);
                if (z < avail) {
                    m |= 1ull << (sgn + z);
                    left -= z + 1;
                    sgn += z + 1;
                } else {
                    left -= avail;
                    sgn += avail;
                    more = sgn >= V;               // else the budget ended inside the run
                }
            }
            spl[p][tid] = m;
        }
        uint32_t lo[32], hi[32];
#pragma unroll
        for (int p = 0; p < 32; ++p) {
            const unsigned long long m = spl[p][tid];
            lo[p] = (uint32_t)m;
            hi[p] = (uint32_t)(m >> 32);
        }
        transpose32(lo);
        if (V > 32) transpose32(hi);
        int32_t iv[V];
#pragma unroll
        for (int r = 0; r < V; ++r) iv[P.p[r]] = unnega(r < 32 ? lo[r] : hi[r < 32 ? 0 : r - 32]);
        xform_inv<DIMS>(iv);
        const float sc = pow2f(max(emax - 23, -126));
#pragma unroll
        for (int i = 0; i < V; ++i) f[i] = __fmul_rn(__int2float_rn(iv[i]), sc);
    }
    // scatter the valid part of the block
    const BlockPos bp = block_pos(G, b);
    const int xs = 4 * bp.bx;
    const bool vec = v.aligned && xs + 3 < v.nx;
    constexpr int ROWS = DIMS == 3 ? 16 : 4;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int z = 4 * bp.bz + (DIMS == 3 ? r / 4 : r);
        const int y = DIMS == 3 ? 4 * bp.by + r % 4 : 0;
        if (z >= v.nz || y >= v.ny) continue;
        float* row = x + (long long)z * v.pz + (long long)y * v.py;
        if (vec) {
            *reinterpret_cast<float4*>(row + xs) = make_float4(f[4 * r], f[4 * r + 1], f[4 * r + 2], f[4 * r + 3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (xs + q < v.nx) row[xs + q] = f[4 * r + q];
        }
    }
}

}  // namespace

long long codec_rate_words(int dims, int nz, int ny, int nx, int rate)
{
    if (rate < 1 || rate > 32) return -1;
    const Geo G = make_geo(dims, nz, ny, nx);
    return HDR + G.nblocks * rate_block_words(dims, rate);
}

cudaError_t codec_rate_compress_dev(const CodecCall& c, cudaStream_t s)
{
    if (c.rate < 1 || c.rate > 32) return cudaErrorInvalidValue;
    const unsigned items = (unsigned)(c.lanes * c.nf);
    const dim3 grd((unsigned)((c.blocks + RT - 1) / RT), items);
    rate_header_kernel<<<dim3(1, items), 32, 0, s>>>(c);
    if (c.dims == 3) rate_enc_kernel<3><<<grd, RT, 0, s>>>(c);
    else rate_enc_kernel<2><<<grd, RT, 0, s>>>(c);
    return cudaGetLastError();
}

cudaError_t codec_rate_decompress_dev(const CodecCall& c, cudaStream_t s)
{
    if (!c.any && (c.rate < 1 || c.rate > 32)) return cudaErrorInvalidValue;
    const dim3 grd((unsigned)((c.blocks + RT - 1) / RT), (unsigned)(c.lanes * c.nf));
    if (c.dims == 3) rate_dec_kernel<3><<<grd, RT, 0, s>>>(c);
    else rate_dec_kernel<2><<<grd, RT, 0, s>>>(c);
    return cudaGetLastError();
}

}  // namespace ckfwi
