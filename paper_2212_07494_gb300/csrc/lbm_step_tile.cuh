// lbm_step_tile.cuh -- K time steps of a D2Q9 lattice in one launch: a block
// advances a TX x TY tile of nodes by K steps with the steps between kept in
// shared memory, so that memory sees one read and one write of the state
// per K steps instead of per step.
//
// Step 1 pulls from memory and computes the tile and a margin of K - 1 nodes
// around it; step s computes the margin K - s from what step s - 1 left in
// shared memory; step K computes the tile itself and stores it.  The margins
// are computed by every tile that needs them, from the same values with the
// same operations, so the result is that of K single steps bit for bit.  In
// shared memory the populations are kept in the storage type (rounded as a
// store to memory rounds them).
//
// A thread takes pairs of neighbouring nodes (x, x + 1): one collision in
// packed FP32, and one 2-element access for every population whose source
// pair starts at an even index (6 of 9 per step; all 9 on the way out).
// Pairs at a wall, at an obstacle or across a periodic x face resolve their
// sources node by node.
//
// What bounds it: on a large FP32 domain memory (36 bytes per node and step
// with K = 2: 90 us for 4096^2) and instructions together (2048^2: DRAM 56 %,
// FMA pipe 62 %, issue 66 % busy; 338 warp instructions per pair and step, 177
// of them on the FMA pipe, margins included); 2-byte storage the instructions
// (FMA pipe 65 %, issue 68 %, DRAM 26 %); a small domain the latency of a
// launch and of a step's dependent instructions.  us per step, one step per launch and
// this kernel, residual and moments included: 4096^2 FP32 183.0 and 114.0
// (1.605x), 4096^2 FP16 101.0 and 99.8, 1001 x 517 with walls 8.90 and 5.21,
// 256 x 128 with obstacles 3.19 and 1.41.
#pragma once
#include "lbm_kernels.cuh"

namespace lbm {

// regions: step s (1 .. K) of a tile covers (TX + 2 (K - s)) x (TY + 2 (K - s)) nodes
template <int TX, int TY, int K> struct TileGeo {
    static constexpr int w(int s) { return TX + 2 * (K - s); }
    static constexpr int h(int s) { return TY + 2 * (K - s); }
    // elements of one population of the buffer that step s writes, and where it
    // starts: odd steps share the first buffer, even ones the second
    static constexpr int plane(int s) { return w(s) * h(s); }
    static constexpr int start(int s) { return (s & 1) ? 0 : 9 * plane(1); }
    static constexpr int elems() { return K == 1 ? 0 : 9 * (plane(1) + (K > 2 ? plane(2) : 0)); }
};

// bits of the populations whose source lies beyond a wall
__device__ __forceinline__ unsigned wall_bits(const TileDom &d, int x, int y) {
    unsigned b = 0u;
    if (!d.per_x) b |= (x == 0 ? 0x122u : 0u) | (x == d.nx - 1 ? 0x0c8u : 0u);   // c_x = +1: 1 5 8; -1: 3 6 7
    if (!d.per_y) b |= (y == 0 ? 0x064u : 0u) | (y == d.ny - 1 ? 0x190u : 0u);   // c_y = +1: 2 5 6; -1: 4 7 8
    return b;
}

// two consecutive elements of the storage type, as the two lanes
template <int ST> __device__ __forceinline__ F2 pair_at(const void *p) {
    if constexpr (ST == ST_F32) {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        return F2::pair(v.x, v.y);
    } else if constexpr (ST == ST_F16) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(p));
        return F2::pair(v.x, v.y);
    } else {
        const unsigned v = *reinterpret_cast<const unsigned *>(p);
        return F2::pair(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
    }
}
template <int ST> __device__ __forceinline__ void pair_to(void *p, F2 v) {
    if constexpr (ST == ST_F32) *reinterpret_cast<float2 *>(p) = make_float2(v.lo(), v.hi());
    else if constexpr (ST == ST_F16) *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(v.lo(), v.hi());
    else *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(v.lo(), v.hi());
}

// memory reads of a tile: through the read-only path, or past L1 where other
// blocks of the same launch write the state (CG)
template <bool CG, typename T> __device__ __forceinline__ T tile_ld(const void *p) {
    if constexpr (CG) return __ldcg(reinterpret_cast<const T *>(p));
    else return __ldg(reinterpret_cast<const T *>(p));
}
template <int ST, bool CG> __device__ __forceinline__ F2 pair_from(const void *p) {
    if constexpr (ST == ST_F32) {
        const float2 v = tile_ld<CG, float2>(p);
        return F2::pair(v.x, v.y);
    } else {
        const unsigned v = tile_ld<CG, unsigned>(p);
        return pair_at<ST>(&v);
    }
}
template <int ST, bool CG> __device__ __forceinline__ float one_from(const void *p) {
    if constexpr (ST == ST_F32) return tile_ld<CG, float>(p);
    else if constexpr (ST == ST_F16) return __half2float(__ushort_as_half(tile_ld<CG, unsigned short>(p)));
    else return __uint_as_float((unsigned)tile_ld<CG, unsigned short>(p) << 16);
}
template <int ST> __device__ __forceinline__ float one_at(const typename Store<ST>::T *p) {
    if constexpr (ST == ST_F32) return *p;
    else if constexpr (ST == ST_F16) return __half2float(*p);
    else return __bfloat162float(*p);
}

// Whether the domain has an obstacle mask: never, always, or when d.links is set
enum { TILE_NO_MASK = 0, TILE_MASK = 1, TILE_ANY_MASK = 2 };

// step S of the tile at (X0, Y0): NT threads (0: blockDim.x), all of them call
// it.  INNER: no node of the tile or its margins, nor any source of theirs,
// lies across a face of the domain, and there is no mask
template <int COLL, int ST, int MASK, bool CG, bool INNER, int TX, int TY, int K, int NT, int S>
__device__ __forceinline__ void tile_step(const TileDom &d, const typename Store<ST>::T *__restrict__ fin,
                                          typename Store<ST>::T *__restrict__ fout, typename Store<ST>::T *sm, int X0,
                                          int Y0) {
    typedef typename Store<ST>::T T;
    typedef TileGeo<TX, TY, K> Geo;
    constexpr int W = Geo::w(S), H = Geo::h(S), M = K - S, PW = W / 2;
    constexpr unsigned ES = sizeof(T);
    const float *g = d.g + (long long)(S - 1) * d.g_step;
    float ugx = 0.f, ugy = 0.f;
    if (d.force_kind == G_UNIFORM) {
        ugx = __ldg(g);
        ugy = __ldg(g + 1);
    }
#pragma unroll 1
    for (int idx = threadIdx.x; idx < PW * H; idx += NT > 0 ? NT : (int)blockDim.x) {
        const int ry = idx / PW, rx = 2 * (idx - ry * PW);
        int x0 = X0 - M + rx, y = Y0 - M + ry;
        int xa = x0, xb = x0 + 1;
        unsigned ba = 0u, bb = 0u;
        if constexpr (!INNER) {
            // coordinates before wrapping; nodes beyond a wall, or further
            // across a periodic face than the tile's own nodes can need, are
            // left out
            if (d.per_y ? y >= d.ny + M : (y < 0 || y >= d.ny)) continue;
            if (d.per_x ? x0 >= d.nx + M : (x0 + 1 < 0 || x0 >= d.nx)) continue;
            if (y < 0) y += d.ny;
            else if (y >= d.ny) y -= d.ny;
            // each node's wrapped x (a node outside a walled row takes its
            // partner's and is not stored)
            if (xa < 0) xa = d.per_x ? xa + d.nx : xb;
            else if (xa >= d.nx) xa -= d.nx;
            if (xb < 0) xb += d.nx;
            else if (xb >= d.nx) xb = d.per_x ? xb - d.nx : xa;
            ba = wall_bits(d, xa, y);
            bb = wall_bits(d, xb, y);
            if (MASK == TILE_MASK || (MASK == TILE_ANY_MASK && d.links)) {
                ba |= __ldg(d.links + y * d.nxp + xa);
                bb |= __ldg(d.links + y * d.nxp + xb);
            }
        }
        F2 G[9];
        if constexpr (S == 1) {
            const int ym = !INNER && y == 0 ? d.ny - 1 : y - 1, yp = !INNER && y == d.ny - 1 ? 0 : y + 1;
            const unsigned row[3] = {(unsigned)(yp * d.nxp) * ES, (unsigned)(y * d.nxp) * ES, (unsigned)(ym * d.nxp) * ES};
            const char *base = reinterpret_cast<const char *>(fin);
            // even pairs: the sources x0 - 1 and x0 + 1 when M is odd, x0 when it is even
            if (INNER || ((ba | bb) == 0u && x0 >= 1 && x0 + 2 < d.nx)) {
                static_for<9>([&](auto I) {
                    constexpr int i = decltype(I)::value, cx = Lat<D2Q9>::cx(i), cy = Lat<D2Q9>::cy(i);
                    const char *q = base + (unsigned)(i * d.plane_bytes + (row[cy + 1] + (unsigned)(x0 - cx) * ES));
                    if constexpr (((M + cx) & 1) == 0) G[gpos<D2Q9>(i)] = pair_from<ST, CG>(q);
                    else G[gpos<D2Q9>(i)] = F2::pair(one_from<ST, CG>(q), one_from<ST, CG>(q + ES));
                });
            } else {
                static_for<9>([&](auto I) {
                    constexpr int i = decltype(I)::value, cx = Lat<D2Q9>::cx(i), cy = Lat<D2Q9>::cy(i);
                    float v[2];
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int x = k ? xb : xa;
                        int sx = x - cx;
                        if (cx == 1 && sx < 0) sx = d.nx - 1;
                        if (cx == -1 && sx >= d.nx) sx = 0;
                        const bool back = ((k ? bb : ba) >> i) & 1u;
                        const unsigned off = back ? row[1] + (unsigned)x * ES : row[cy + 1] + (unsigned)sx * ES;
                        v[k] = one_from<ST, CG>(base + (unsigned)((back && i != 0 ? opp<D2Q9>(i) : i) * d.plane_bytes + off));
                    }
                    G[gpos<D2Q9>(i)] = F2::pair(v[0], v[1]);
                });
            }
        } else {
            constexpr int PL = Geo::plane(S - 1), PWD = Geo::w(S - 1);
            const T *own = sm + Geo::start(S - 1) + (ry + 1) * PWD + rx + 1;
            if (INNER || (ba | bb) == 0u) {
                static_for<9>([&](auto I) {
                    constexpr int i = decltype(I)::value, cx = Lat<D2Q9>::cx(i), cy = Lat<D2Q9>::cy(i);
                    const T *q = own + (i * PL - cy * PWD - cx);
                    if constexpr (cx != 0) G[gpos<D2Q9>(i)] = pair_at<ST>(q);
                    else G[gpos<D2Q9>(i)] = F2::pair(one_at<ST>(q), one_at<ST>(q + 1));
                });
            } else {
                static_for<9>([&](auto I) {
                    constexpr int i = decltype(I)::value, cx = Lat<D2Q9>::cx(i), cy = Lat<D2Q9>::cy(i);
                    constexpr int nb = i * PL - cy * PWD - cx, back = (i ? opp<D2Q9>(i) : 0) * PL;
                    G[gpos<D2Q9>(i)] = F2::pair(one_at<ST>(own + (((ba >> i) & 1u) ? back : nb)),
                                                one_at<ST>(own + 1 + (((bb >> i) & 1u) ? back : nb)));
                });
            }
        }
        F2 gx = F2(ugx), gy = F2(ugy);
        if (d.force_kind == G_ROWS) {
            gx = F2(__ldg(g + 2 * y));
            gy = F2(__ldg(g + 2 * y + 1));
        } else if (d.force_kind == G_FIELD) {
            const float *q = g + (long long)y * d.nxp;
            gx = F2::pair(__ldg(q + xa), __ldg(q + xb));
            gy = F2::pair(__ldg(q + d.g_plane + xa), __ldg(q + d.g_plane + xb));
        }
        collide_any<D2Q9, COLL>(G, gx, gy, F2(0.0f), F2(d.om2), F2(d.om3), F2(d.om4), F2(d.omb));
        if constexpr (S < K) {
            T *q = sm + Geo::start(S) + ry * W + rx;
            static_for<9>([&](auto I) {
                constexpr int i = decltype(I)::value;
                pair_to<ST>(q + i * Geo::plane(S), G[gpos<D2Q9>(i)]);
            });
        } else {
            char *out = reinterpret_cast<char *>(fout);
            const unsigned q = ((unsigned)(y * d.nxp) + (unsigned)x0) * ES;
            // bit 0: a solid node
            const bool sa = INNER || (ba & 1u) == 0u, sb = INNER || (x0 + 1 < d.nx && (bb & 1u) == 0u);
            if (sa && sb) {
                static_for<9>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    pair_to<ST>(out + (unsigned)(q + i * d.plane_bytes), G[gpos<D2Q9>(i)]);
                });
            } else {
                static_for<9>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    T *o = reinterpret_cast<T *>(out + (unsigned)(q + i * d.plane_bytes));
                    if (sa) Store<ST>::st(o, G[gpos<D2Q9>(i)].lo());
                    if (sb) Store<ST>::st(o + 1, G[gpos<D2Q9>(i)].hi());
                });
            }
        }
    }
}

// all K steps of the tile at (X0, Y0)
template <int COLL, int ST, int MASK, bool CG, int TX, int TY, int K, int NT>
__device__ __forceinline__ void tile_steps(const TileDom &d, const typename Store<ST>::T *__restrict__ fin,
                                           typename Store<ST>::T *__restrict__ fout, typename Store<ST>::T *sm, int X0,
                                           int Y0) {
    auto run = [&](auto inner) {
        static_for<K>([&](auto I) {
            constexpr int S = decltype(I)::value + 1;
            if constexpr (S > 1) __syncthreads();
            tile_step<COLL, ST, MASK, CG, decltype(inner)::value != 0, TX, TY, K, NT, S>(d, fin, fout, sm, X0, Y0);
        });
    };
    if constexpr (MASK != TILE_MASK) {
        // most tiles of a large domain: the whole block takes the path
        // without wraps, walls and limits
        if ((MASK == TILE_NO_MASK || !d.links) && X0 >= K && Y0 >= K && X0 + TX + K <= d.nx && Y0 + TY + K <= d.ny) {
            run(Idx<1>{});
            return;
        }
    }
    run(Idx<0>{});
}

// MINB blocks of NT threads per SM cap the registers at 64
template <int COLL, int ST, int MASK, int TX, int TY, int K, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_step_tile(const __grid_constant__ TileDom d,
                                                        const typename Store<ST>::T *__restrict__ fin,
                                                        typename Store<ST>::T *__restrict__ fout) {
    extern __shared__ __align__(16) unsigned char tile_smem[];
    tile_steps<COLL, ST, MASK, false, TX, TY, K, NT>(d, fin, fout, reinterpret_cast<typename Store<ST>::T *>(tile_smem),
                                                     blockIdx.x * TX, blockIdx.y * TY);
}

// host launcher of one storage type and mask flag: K = 4 or 2 steps
template <int ST, bool MASK> struct TileDispatch {
    typedef typename Store<ST>::T T;
    template <int COLL, int TX, int TY, int K, int NT, int MINB>
    static cudaError_t go(const TileDom &d, const void *fin, void *fout, cudaStream_t s) {
        constexpr size_t smem = TileGeo<TX, TY, K>::elems() * sizeof(T);
        static_assert(smem <= 48 * 1024, "within the default dynamic shared memory");
        const dim3 grid((unsigned)((d.nx + TX - 1) / TX), (unsigned)((d.ny + TY - 1) / TY));
        k_step_tile<COLL, ST, MASK ? TILE_MASK : TILE_NO_MASK, TX, TY, K, NT, MINB><<<grid, NT, smem, s>>>(d, (const T *)fin, (T *)fout);
        return cudaGetLastError();
    }
    template <int COLL>
    static cudaError_t by_steps(int K, const TileDom &d, const void *fin, void *fout, cudaStream_t s) {
        // Tile shapes measured on GB300, us per step (F32 unless stated).
        // Two steps: 32 x 8, 192 threads: 4096^2 109.0 (32 x 16 109.9, 64 x 16 114, 16 x 8 114), 1024^2 7.4,
        // 512^2 2.8; in 2-byte storage 30 x 14, 128 threads: 93.7 (32 x 16 99.5, 64 x 32 94.0).  Four steps:
        // 16 x 16, 256 threads: 256 x 128 1.15, 400 x 300 1.82 (two steps 1.95), 512^2 2.95 (two steps 2.82).
        if (K == 4) return go<COLL, 16, 16, 4, 256, 4>(d, fin, fout, s);
        if (K != 2) return cudaErrorInvalidValue;
        if constexpr (sizeof(T) == 4) return go<COLL, 32, 8, 2, 192, 5>(d, fin, fout, s);
        else return go<COLL, 30, 14, 2, 128, 8>(d, fin, fout, s);
    }
    static cudaError_t step(int coll, int K, const TileDom &d, const void *fin, void *fout, cudaStream_t s) {
        switch (coll) {
        case SMRT:
            // the trimmed collision under k_step's conditions
            if (d.trim) return by_steps<SMRT_TRIM>(K, d, fin, fout, s);
            return by_steps<SMRT>(K, d, fin, fout, s);
        case SMRT_FNEQ: return by_steps<SMRT_FNEQ>(K, d, fin, fout, s);
        case MRT_RAW: return by_steps<MRT_RAW>(K, d, fin, fout, s);
        case BGK: return by_steps<BGK>(K, d, fin, fout, s);
        }
        return cudaErrorInvalidValue;
    }
};

}  // namespace lbm
