// k_generic.cu -- pass kernels whose radix list is data: any 2*3*5-smooth line
// length up to 4096, the 2D slab pass of the slab-pencil decomposition for
// slabs that fit in one block's shared memory, the identity probe of a pass
// geometry, and the copy pass.
#include "fix64.cuh"
#include "pass_kernels.cuh"
#include "runtime_stages.cuh"

namespace fft3 {

// ------------------------------------------------------------ k_pass_g -- //
// One tile of `lpt` lines staged through shared memory (whichever mapping
// keeps the global accesses coalesced), the runtime radix stages, the tile
// stored back.
struct TileG {
    int64_t nval;     // lines of this tile inside the array
    int64_t ib, ob;   // offsets of the tile's first line in the input and the output
};
__device__ __forceinline__ TileG tile_g(const PassArgs &a, int64_t tile)
{
    const TileId id = decode_tile(tile, a.tiles_c, a.g.A, a.lpt);
    return TileG{min((int64_t)a.lpt, a.g.C - id.c0), id.c0 * a.g.ic + id.a * a.g.ia + id.b * a.g.ib,
                 id.c0 * a.g.oc + id.a * a.g.oa + id.b * a.g.ob};
}
template <class C>
__device__ __forceinline__ void tile_g_load(const PassArgs &a, const TileG &t, const C *in, C *buf, int n, int P)
{
    const bool lines = a.g.ij == 1, conj = a.conj != 0;
    for (int e = threadIdx.x; e < a.lpt * n; e += blockDim.x) {
        int l, j;
        if (lines) { l = e / n; j = e - l * n; }
        else { l = e % a.lpt; j = e / a.lpt; }
        C v = Cx<C>::make(0, 0);
        if (l < t.nval)
            v = in[t.ib + l * a.g.ic + geom_in_elem(a.g, j)];
        buf[l * P + padpos(j)] = conj ? cconj(v) : v;
    }
}
// value(l, slot): the result at shared slot `slot` of line l.
template <class C, class Value>
__device__ __forceinline__ void tile_g_store(const PassArgs &a, const TileG &t, C *out, int n, int P, const Value &value)
{
    const bool lines = a.g.ok == 1, conj = a.conj != 0;
    for (int e = threadIdx.x; e < a.lpt * n; e += blockDim.x) {
        int l, k;
        if (lines) { l = e / n; k = e - l * n; }
        else { l = e % a.lpt; k = e / a.lpt; }
        if (l < t.nval) {
            const C v = value(l, l * P + padpos(k));
            out[t.ob + l * a.g.oc + geom_out_elem(a.g, k)] = conj ? cconj(v) : v;
        }
    }
}

__global__ void k_pass_g(PassArgs a)
{
    extern __shared__ __align__(16) unsigned char g_smem_raw[];
    float2 *tw = reinterpret_cast<float2 *>(g_smem_raw);
    const LineRt &L = a.L[0];
    const int P = line_pitch(L.n);
    float2 *b0 = tw + tw_slots(a.tw_len), *b1 = b0 + a.lpt * P;
    load_twiddles(tw, a.tw, a.tw_len);
    pdl_wait();
    for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        __syncthreads();
        const TileG t = tile_g(a, tile);
        tile_g_load(a, t, a.in, b0, L.n, P);
        __syncthreads();
        const float2 *res = run_stages_lines(L, a.lpt, P, b0, b1, tw + L.tw_off);
        tile_g_store(a, t, a.out, L.n, P, [&](int, int slot) { return res[slot]; });
    }
}

// ---------------------------------------------------------- k_pass_g64 -- //
// The complex128 path: the same tile in 64-bit block fixed point (fix64.cuh),
// every line normalised after each of its stages.  Per line the block keeps
// its largest magnitude words, the least of its first-stage butterflies', the sum of
// its shifts and three rotating words for the normalisation (stage s fills slot s % 3, reads the one before and clears
// the one after).  A tile with a line the integers do not take runs the FP64
// stages on the same buffers, its twiddles read from global memory.
struct FixLineState {
    FixMag *line;  // [lpt]
    unsigned *least; // [lpt], complemented
    int *up;       // [lpt]; during the scan: whether a first-stage butterfly is all zeros
    unsigned *nrm; // [3][lpt]
};

template <int R>
__device__ __forceinline__ void stage_fix_rt(const LineRt &L, int NS, int t, const fix2 *src, fix2 *dst,
                                             const root62 *tw, bool first, int emax, int up, unsigned *acc_out)
{
    const int NB = L.n / R;
    unsigned acc = 0;
    for (int q = t; q < NB; q += L.T) {
        fix2 v[R];
        const int k = q % NS;
        if (first) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const double2 x = reinterpret_cast<const double2 *>(src)[padpos(q + r * NB)];
                v[r] = fix2{to_fix<true>(x.x, emax), to_fix<true>(x.y, emax)};
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
                v[r] = shl(src[padpos(q + r * NB)], up);
            v[0] = quarter<true>(v[0]);
#pragma unroll
            for (int r = 1; r < R; ++r)
                v[r] = cmul62(v[r], tw[(r - 1) * NS + k]);
        }
        BflyFix<R, true>::run(v);
        const int base = (q / NS) * NS * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            dst[padpos(base + r * NS)] = v[r];
            acc |= norm_word(v[r].x) | norm_word(v[r].y);
        }
    }
    atomicOr(acc_out, acc);
}

__device__ __forceinline__ int fix_scale_rt(int R) { return R == 16 || R == 8 ? 2 : R == 5 ? 1 : 0; }

__device__ __forceinline__ fix2 *run_stages_fix(const LineRt &L, int lpt, int P, fix2 *A, fix2 *B, const root62 *tw,
                                                const FixLineState &st)
{
    const int nteams = blockDim.x / L.T;
    const int team = threadIdx.x / L.T, t = threadIdx.x - team * L.T;
    fix2 *cur = A, *nxt = B;
    int NS = 1, off = 0;
    for (int s = 0; s < L.nst; ++s) {
        const int R = L.rad[s];
        unsigned *fill = st.nrm + (s % 3) * lpt, *prev = st.nrm + ((s + 2) % 3) * lpt,
                 *clear = st.nrm + ((s + 1) % 3) * lpt;
        if (team < nteams)
            for (int l = team; l < lpt; l += nteams) {
                const fix2 *src = cur + l * P;
                fix2 *dst = nxt + l * P;
                const int emax = fix_emax(mag_all(st.line[l]));
                const int up = s ? norm_shift(prev[l]) : 0;
                if (t == 0) {
                    clear[l] = 0;
                    st.up[l] = s ? st.up[l] + up : 0;
                }
                switch (R) {
                case 2: stage_fix_rt<2>(L, NS, t, src, dst, tw + off, s == 0, emax, up, fill + l); break;
                case 3: stage_fix_rt<3>(L, NS, t, src, dst, tw + off, s == 0, emax, up, fill + l); break;
                case 4: stage_fix_rt<4>(L, NS, t, src, dst, tw + off, s == 0, emax, up, fill + l); break;
                case 5: stage_fix_rt<5>(L, NS, t, src, dst, tw + off, s == 0, emax, up, fill + l); break;
                case 8: stage_fix_rt<8>(L, NS, t, src, dst, tw + off, s == 0, emax, up, fill + l); break;
                case 16: stage_fix_rt<16>(L, NS, t, src, dst, tw + off, s == 0, emax, up, fill + l); break;
                default: break;
                }
            }
        __syncthreads();
        off += (R - 1) * NS;
        NS *= R;
        fix2 *x = cur;
        cur = nxt;
        nxt = x;
    }
    return cur;
}

// FP64 stages of a loaded tile (b0) and its store.
__device__ __noinline__ void tile_g64_fp64(const PassArgs &a, const TileG &t, double2 *b0, double2 *b1, int P)
{
    const LineRt &L = a.L[0];
    const double2 *res =
        run_stages_lines(L, a.lpt, P, b0, b1, reinterpret_cast<const double2 *>(a.tw) + L.tw_off);
    tile_g_store(a, t, reinterpret_cast<double2 *>(a.out), L.n, P, [&](int, int slot) { return res[slot]; });
}

__global__ void __launch_bounds__(512) k_pass_g64(PassArgs a) // kMaxThreadsG64
{
    extern __shared__ __align__(16) unsigned char g_smem_raw[];
    const LineRt &L = a.L[0];
    const int n = L.n, P = line_pitch(n), lpt = a.lpt;
    root62 *tw = reinterpret_cast<root62 *>(g_smem_raw);
    fix2 *b0 = reinterpret_cast<fix2 *>(tw + tw_slots(a.tw_len)), *b1 = b0 + lpt * P;
    unsigned *words = reinterpret_cast<unsigned *>(b1 + lpt * P);
    const FixLineState st{reinterpret_cast<FixMag *>(words), words + 2 * lpt, reinterpret_cast<int *>(words + 3 * lpt),
                          words + 4 * lpt};
    const root62 *twg = reinterpret_cast<const root62 *>(a.tw_fix);
    for (int i = threadIdx.x; i < a.tw_len; i += blockDim.x)
        tw[i] = twg[i];
    pdl_wait();
    int scale = 0, exact = fix_exact_bits(0); // powers of two the stages scale down by; least fix_exact_bits
    for (int s = 0; s < L.nst; ++s) {
        scale += fix_scale_rt(L.rad[s]) + (s ? 2 : 0);
        exact = min(exact, fix_exact_bits(fix_scale_rt(L.rad[s])));
    }
    const int nteams = blockDim.x / L.T, team = threadIdx.x / L.T, t = threadIdx.x - team * L.T;
    const int R0 = L.nst ? L.rad[0] : 1, NB0 = n / R0; // first-stage butterflies
    for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        __syncthreads();
        const TileG tg = tile_g(a, tile);
        for (int i = threadIdx.x; i < kFix64LineWords * lpt; i += blockDim.x)
            words[i] = 0;
        tile_g_load(a, tg, reinterpret_cast<const double2 *>(a.in), reinterpret_cast<double2 *>(b0), n, P);
        __syncthreads();
        if (team < nteams)
            for (int l = team; l < lpt; l += nteams) {
                FixScan scan;
                for (int q = t; q < NB0; q += L.T) {
                    FixMag m{0u, 0u};
                    for (int r = 0; r < R0; ++r)
                        mag_max(m, reinterpret_cast<const double2 *>(b0)[l * P + padpos(q + r * NB0)]);
                    scan.add(m);
                }
                atomicMax(&st.line[l].re, scan.line.re);
                atomicMax(&st.line[l].im, scan.line.im);
                atomicMax(st.least + l, ~scan.least);
                if (scan.zeros || L.nst == 1)
                    st.up[l] = 1;
            }
        __syncthreads();
        bool bad = false;
        for (int l = threadIdx.x; l < lpt; l += blockDim.x)
            bad = bad || !fix_ok(FixScan{st.line[l], ~st.least[l], st.up[l] != 0}, fix_strict(n, R0), exact);
        if (__syncthreads_or(bad)) {
            tile_g64_fp64(a, tg, reinterpret_cast<double2 *>(b0), reinterpret_cast<double2 *>(b1), P);
            continue;
        }
        const fix2 *res = run_stages_fix(L, lpt, P, b0, b1, tw + L.tw_off, st);
        const bool none = L.nst == 0; // one-point lines move their values as they are
        tile_g_store(a, tg, reinterpret_cast<double2 *>(a.out), n, P, [&](int l, int slot) {
            const fix2 v = res[slot];
            if (none)
                return reinterpret_cast<const double2 *>(res)[slot];
            const int sh = fix_emax(mag_all(st.line[l])) - 1081 + scale - st.up[l];
            return make_double2(from_fix(v.x, sh), from_fix(v.y, sh));
        });
    }
}

// -------------------------------------------------------------- k_slab -- //
// One n0 x n1 slab per tile, held in shared memory: x lines (rows, length n0)
// then y lines (columns, length n1), ping-ponging between two padded copies.
__global__ void k_slab(PassArgs a)
{
    extern __shared__ float2 smem[];
    const LineRt &X = a.L[0];
    const LineRt &Y = a.L[1];
    const int n0 = X.n, n1 = Y.n;
    const int P = line_pitch(n0);
    float2 *tw = smem;
    float2 *b0 = smem + tw_slots(a.tw_len);
    float2 *b1 = b0 + n1 * P;
    load_twiddles(tw, a.tw, a.tw_len);
    pdl_wait();
    const bool conj = a.conj != 0;
    const int nel = n0 * n1;
    for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        __syncthreads();
        const int64_t sa = tile % a.g.A, sb = tile / a.g.A;
        const float2 *ib = a.in + sa * a.g.ia + sb * a.g.ib;
        float2 *ob = a.out + sa * a.g.oa + sb * a.g.ob;
        for (int e = threadIdx.x; e < nel; e += blockDim.x) {
            const int row = e / n0, col = e - row * n0;
            const float2 v = ib[e];
            b0[row * P + padpos(col)] = conj ? cconj(v) : v;
        }
        __syncthreads();
        float2 *r1 = run_stages_lines(X, n1, P, b0, b1, tw + X.tw_off);
        float2 *o1 = (r1 == b0) ? b1 : b0;
        float2 *r2 = run_stages_cols(Y, n0, P, r1, o1, tw + Y.tw_off);
        for (int e = threadIdx.x; e < nel; e += blockDim.x) {
            const int row = e / n0, col = e - row * n0;
            const float2 v = r2[row * P + padpos(col)];
            ob[e] = conj ? cconj(v) : v;
        }
    }
}

// ------------------------------------------------------- k_probe_pass -- //
// Identity line transform on the pass geometry: element j of every input
// line is written to element j of its output line.
__global__ void k_probe_pass(PassArgs a)
{
    const int64_t n = a.L[0].n;
    const int64_t total = n * a.g.C * a.g.A * a.g.B;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = e % n, r = e / n;
        const int64_t c = r % a.g.C;
        r /= a.g.C;
        const int64_t aa = r % a.g.A, b = r / a.g.A;
        a.out[geom_out_elem(a.g, j) + c * a.g.oc + aa * a.g.oa + b * a.g.ob] =
            a.in[geom_in_elem(a.g, j) + c * a.g.ic + aa * a.g.ia + b * a.g.ib];
    }
}

// --------------------------------------------------------------- k_copy -- //
__global__ void k_copy(const float2 *in, float2 *out, int64_t total)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = in[i];
}

} // namespace fft3
