// pps_trunc.cuh -- the truncated race: top-k, then top-p, then the race over
// the surviving tokens.  Included by pps_race.cu, whose Philox, lists, row
// finalisation and tree walk it reuses (one translation unit).
//
// Truncation (the experiments sample with top-k = 50, top-p = 1, Sec. 6; a
// truncated distribution has a support of at most k tokens, Sec. 4.2) sets
// P = 0, i.e. E/P = +inf, outside the kept set S, so the race of the truncated
// distribution is argmin over S of s = ln E - l/T (the renormalisation of P on
// S does not move the argmin).  The set: every token whose logit is >= l_(k),
// the k-th largest usable logit (all ties of l_(k) are kept); then, if
// top_p < 1, whole groups of equal logits are removed in ascending order while
// the running probability mass (softmax(l/T) over the top-k set, summed token
// by token in ascending order) is <= 1 - top_p; the top group always stays.
//
// Work per row.  The streaming pass only finds S: one max of the iteration's
// logits per lane (packed bf16x2 max for bf16 rows) against the warp's
// threshold, a lower bound of l_(k).  No Philox word is needed for a token
// outside S, so the pass is bound by HBM rather than by the multiply pipe.
// Vectors with a logit at or over the threshold are queued and their tokens
// appended to a buffer; when it fills it is compacted to the tokens that can
// still be in S, which raises the threshold.  Tokens below the threshold are
// below l_(k) and can be dropped for good; a token tied with it that did not fit
// is recorded in `dropmax`, and if one ties with l_(k) the buffer does not hold
// the whole tie group: the row is then finished by a counting pass (for top-p) and, when
// the tie group stays in S, by the exact fp32 race of pps_race.cu over the
// tokens with logit >= l_(k).  Otherwise the finishing warp keys the <= 64
// surviving tokens with the race's fp32 key, keeps the smallest and hands
// them to finalize_row, which re-keys in fp64 (s = ln E - l/T) every pair closer
// than the fp32 error bounds, so the row is emitted exactly like the
// untruncated race; a row whose K-th key is that close to a key left out takes
// the fp64 keys of all of S (finish_crowded).
//
// A step of the benchmark's tree (top-k 50: 1.21 GB of logits) takes 266 us =
// 4.6 TB/s, 290 when every row's threshold climbed from the first iteration's and S
// was sorted; one sequence 263 -> 88 us; 16720 rows of V = 5717 736 -> 248 us.  It is
// bound by HBM (0.78 of the measured copy rate inside the launch; the sample, 6.4% of a row,
// is read twice) and by the finish of the last rows, about 12 us a launch.

#ifndef PPS_TRUNC_UNITS
#define PPS_TRUNC_UNITS 8  // 16-byte vectors per lane per iteration of the top-k scan (even)
#endif
#ifndef PPS_TRUNC_EAGER
#define PPS_TRUNC_EAGER 192  // buffered candidates at which a queue flush also compacts (at 96: 282 us instead of 266)
#endif
#ifndef PPS_TRUNC_MIN_BLOCKS
#define PPS_TRUNC_MIN_BLOCKS 20
#endif
#ifndef PPS_TRUNC_SEG_CAP
#define PPS_TRUNC_SEG_CAP 16
#endif
constexpr int kTruncSegCap = PPS_TRUNC_SEG_CAP;  // at most this many warps per row (one sequence: 8 98 us, 16 87, 32 93)
#ifndef PPS_TRUNC_MIN_VECS
#define PPS_TRUNC_MIN_VECS 512
#endif
// a row is not cut finer: a step of 132 rows of V = 7338 took 66 us with 256 and 58 with 512; lists of 64
// rows of 512, 1024 and 2048 vectors take 23, 23.5 and 27.4 us with 256, 19.3, 25.9 and 26.5 with 512, and
// 19.3, 27.6 and 33.6 with 1024
constexpr int64_t kTruncMinVecs = PPS_TRUNC_MIN_VECS;
constexpr int kTruncRounds = 8;  // kept lists up to this long are selected by argmin rounds

// ---------------------------------------------------------------- top lists
// A top list holds up to 64 entries (v, i) in "top order": logit descending,
// then token ascending (only top-p needs the order).  Entry m sits in lane m
// (av, ai) for m < 32 and in lane m - 32 (bv, bi) otherwise; empty entries are
// (-inf, INT_MAX).  NaN and -inf logits never enter.

__device__ __forceinline__ bool top_before(float av, int ai, float bv, int bi) {
    return av > bv || (av == bv && ai < bi);
}

// bitonic sort of one entry per lane into top order (lane 0 first)
__device__ __forceinline__ void top_sort(float& v, int& i, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const float ov = __shfl_xor_sync(FULL, v, stride);
            const int oi = __shfl_xor_sync(FULL, i, stride);
            const bool up = (lane & size) == 0 || size == 32;
            const bool lower = (lane & stride) == 0;
            const bool o_first = top_before(ov, oi, v, i);
            const bool take = (lower == up) ? o_first : (!o_first && !(ov == v && oi == i));
            if (take) {
                v = ov;
                i = oi;
            }
        }
    }
}

// bitonic half-cleaner pass over a bitonic sequence (one entry per lane)
__device__ __forceinline__ void top_clean(float& v, int& i, int lane) {
#pragma unroll
    for (int stride = 16; stride > 0; stride >>= 1) {
        const float ov = __shfl_xor_sync(FULL, v, stride);
        const int oi = __shfl_xor_sync(FULL, i, stride);
        const bool lower = (lane & stride) == 0;
        const bool o_first = top_before(ov, oi, v, i);
        if (lower ? o_first : (!o_first && !(ov == v && oi == i))) {
            v = ov;
            i = oi;
        }
    }
}

// two sorted lists x, y -> h = the first 32 of their union, l = the last 32, both sorted
__device__ __forceinline__ void top_merge(float xv, int xi, float yv, int yi, float& hv, int& hi, float& lv, int& li,
                                          int lane) {
    const float rv = __shfl_sync(FULL, yv, 31 - lane);
    const int ri = __shfl_sync(FULL, yi, 31 - lane);
    const bool xf = top_before(xv, xi, rv, ri);
    hv = xf ? xv : rv;
    hi = xf ? xi : ri;
    lv = xf ? rv : xv;
    li = xf ? ri : xi;
    top_clean(hv, hi, lane);
    top_clean(lv, li, lane);
}

// the buffer's entries in top order: entries lane and lane + 32
struct TopList {
    float av, bv;
    int ai, bi;
};

// ---------------------------------------------------------------- vector helpers

// any half of the bf16 pair m >= the bf16 pair t2 (NaN halves compare false)
__device__ __forceinline__ bool bf2_any_ge(uint32_t m, uint32_t t2) {
    uint32_t r;
    asm("{\n\t.reg .pred p, q;\n\t"
        "setp.ge.bf16x2 p|q, %1, %2;\n\t"
        "or.pred p, p, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(m), "r"(t2));
    return r != 0;
}

// largest usable logit of vectors d[k0 .. k0+n) (NaN ignored, -inf if none)
template <int DT, int N>
__device__ __forceinline__ float vecs_max(const uint4 (&d)[N], int k0, int n) {
    float r = -kInf;
#pragma unroll
    for (int k = k0; k < k0 + n; ++k) {
        if constexpr (DT == 1) {
            const uint32_t m = bf2_max(bf2_max(d[k].x, d[k].y), bf2_max(d[k].z, d[k].w));
            r = fmaxf(r, fmaxf(bf16_lo(m), bf16_hi(m)));
        } else {
            r = fmaxf(r, fmaxf(fmaxf(__uint_as_float(d[k].x), __uint_as_float(d[k].y)),
                               fmaxf(__uint_as_float(d[k].z), __uint_as_float(d[k].w))));
        }
    }
    return r;  // fmaxf returns the non-NaN operand
}

// ---------------------------------------------------------------- the top-k scan

// order-preserving unsigned key of a float (NaN never reaches it)
__device__ __forceinline__ uint32_t order_key(float x) {
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_order_key(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// The k-th largest of the warp's 32 x N order keys, bit by bit (bf16 values: the
// high 16 bits decide, the low ones are all 0, or all 1 below zero).  At least k
// of them are not 0.
template <int DT, int N>
__device__ __forceinline__ uint32_t kth_order_key(const uint32_t (&key)[N], int k) {
    uint32_t res = 0;
#pragma unroll 1
    for (int b = 31; b >= (DT == 1 ? 16 : 0); --b) {
        const uint32_t cand = res | (1u << b);
        int n = 0;
#pragma unroll
        for (int j = 0; j < N; ++j) n += key[j] >= cand;
        if (__reduce_add_sync(FULL, (unsigned)n) >= (unsigned)k) res = cand;
    }
    return DT == 1 && !(res & 0x80000000u) ? res | 0xffffu : res;
}

// Threshold for an empty buffer, from the first iteration's vectors: the
// k-th largest of the 32 x NV per-vector maxima (bitwise search on order
// keys).  They are maxima of distinct vectors of the segment, so at least k
// of its tokens reach it and l_(k) >= it.
template <int DT>
__device__ __forceinline__ float seed_thr(const uint4 (&d)[PPS_TRUNC_UNITS], int k) {
    constexpr int NV = PPS_TRUNC_UNITS;
    uint32_t key[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) key[j] = order_key(vecs_max<DT>(d, j, 1));
    return from_order_key(kth_order_key<DT, NV>(key, k));
}

// A guess of l_(k) for a long segment, from 32 sampled chunks of 32 vectors
// spread evenly over [v0, vend) (`row`: the interior's start): the j-th largest
// of the 32 chunk maxima, j three deviations and three above the number of
// top-k tokens expected in the sample.  With it the scan buffers about
// j / f tokens of a segment sampled at f = 32 chunks / all chunks (200 of 128256, k =
// 50) and hardly ever compacts; the threshold the first iteration proves
// lets through ~1000 and compacts every 46 (a step of the benchmark's tree 289 -> 263 us).  It is a guess: topk_segment checks
// that k tokens reached it.  One maximum per chunk keeps a cluster of large
// logits (a vocabulary sorted by frequency) from raising it.  What it costs: a row
// in descending order, whose first iteration holds the top k, pays for the sample alone (1024
// rows of V = 128256 bf16 66 -> 73 us, of random rows 101 -> 87), and a row with its largest
// logits all in the sampled chunks (a random one: once in 10^4) is scanned twice (101 -> 128 us).
// Sixteen chunks loaded together instead of eight spill (265 -> 270 us).
constexpr int kSampleChunks = 32;
// vectors from which a segment takes a guess: 3040 rows of V = 49160 bf16 (6145 vectors) 88.3 -> 85.0 us with
// it, of V = 72000 109.5 -> 95.0; rows of 4500 vectors would gain too (76.9 -> 71.8 us), segments of
// 3072 from k = 10 on some (51.7 -> 47.2) and from k = 50 on not (67.2 -> 69.4)
constexpr int64_t kSampleMin = 32 * 192;

template <int DT>
__device__ __noinline__ float guess_thr(const char* row, int64_t v0, int64_t vend, int k) {
    constexpr int B = 8;  // chunks loaded together
    const int lane = threadIdx.x & 31;
    const int64_t chunks = (vend - v0) / 32;
    const uint4* p = reinterpret_cast<const uint4*>(row) + v0 + lane;
    uint32_t mine = 0;  // lane c: order key of chunk c's largest logit
#pragma unroll 1
    for (int c0 = 0; c0 < kSampleChunks; c0 += B) {
        uint4 d[B];
#pragma unroll
        for (int j = 0; j < B; ++j) d[j] = ldg_stream(p + (chunks * (c0 + j) / kSampleChunks) * 32);
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const uint32_t m = __reduce_max_sync(FULL, order_key(vecs_max<DT>(d, j, 1)));
            if (lane == c0 + j) mine = m;
        }
    }
    const float x = (float)(kSampleChunks * k) / (float)chunks;
    const int j = (int)(x + 3.0f * sqrtf(x) + 4.0f);  // < 32 for k <= kTopMax and kSampleMin vectors
    uint32_t res = 0;
    for (int b = 31; b >= 0; --b) {
        const uint32_t cand = res | (1u << b);
        if (__popc(__ballot_sync(FULL, mine >= cand)) >= j) res = cand;
    }
    return from_order_key(res);
}

// The scan appends every token the segment may still need to a per-warp
// buffer in shared memory and raises the threshold only when the buffer
// fills: then the k-th largest logit t of the buffer becomes the threshold
// and the buffer keeps the tokens above t and as many tied with t as the
// 64-entry list holds (dropmax records the rest).  Appending is cheap; the
// exact selection runs a few times per segment.
constexpr int kCandCap = 256;

struct CandState {
    float thr;      // lower bound of l_(k): tokens below it cannot be in S
    float dropmax;  // largest logit dropped from the buffer (-inf: none)
    int n;          // buffered entries
    // A token can still change S: above the threshold, or tied with it while no
    // token of that logit has been dropped yet (once one has, the row's tie
    // group at that logit, if it is l_(k), overflows whatever else arrives).
    __device__ __forceinline__ bool wants(float x) const {
        return x > -kInf && (x > thr || (x == thr && dropmax < thr));
    }
};

template <int DT>
__device__ __noinline__ CandState cand_compact(CandState C, float* sv, int* si, int k) {
    constexpr int PER = kCandCap / 32;
    const int lane = threadIdx.x & 31;
    if (C.n < k) return C;
    float v[PER];
    int ix[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int q = j * 32 + lane;
        v[j] = q < C.n ? sv[q] : -kInf;
        ix[j] = q < C.n ? si[q] : INT_MAX;
    }
    __syncwarp();
    // t = the k-th largest buffered logit
    uint32_t ok[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) ok[j] = v[j] > -kInf ? order_key(v[j]) : 0u;
    const uint32_t res = kth_order_key<DT, PER>(ok, k);
    const float t = from_order_key(res);
    int ng = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) ng += v[j] > t;
    const int g = (int)__reduce_add_sync(FULL, (unsigned)ng);  // < k
    const int room = kTopMax - g;
    int wg = 0, wt = 0;  // written so far (greater, tied)
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const bool gt = v[j] > t, eq = v[j] == t;
        const unsigned mg = __ballot_sync(FULL, gt), me = __ballot_sync(FULL, eq);
        const unsigned below = (1u << lane) - 1u;
        if (gt) {
            const int o = wg + __popc(mg & below);
            sv[o] = v[j];
            si[o] = ix[j];
        }
        if (eq) {
            const int o = wt + __popc(me & below);
            if (o < room) {
                sv[g + o] = v[j];
                si[g + o] = ix[j];
            }
        }
        wg += __popc(mg);
        wt += __popc(me);
    }
    __syncwarp();
    if (wt > room) C.dropmax = fmaxf(C.dropmax, t);
    C.n = g + min(wt, room);
    C.thr = fmaxf(C.thr, t);
    return C;
}

// the buffer (n <= 64 entries) as a sorted top list
__device__ __noinline__ TopList cand_to_list(int n, const float* sv, const int* si) {
    const int lane = threadIdx.x & 31;
    TopList L;
    float av = lane < n ? sv[lane] : -kInf, bv = 32 + lane < n ? sv[32 + lane] : -kInf;
    int ai = lane < n ? si[lane] : INT_MAX, bi = 32 + lane < n ? si[32 + lane] : INT_MAX;
    top_sort(av, ai, lane);
    top_sort(bv, bi, lane);
    top_merge(av, ai, bv, bi, L.av, L.ai, L.bv, L.bi, lane);
    return L;
}

// Append each lane's token (x, i) that is wanted (x = -inf: none); the buffer is compacted when it runs over.
template <int DT>
__device__ __forceinline__ void cand_push(CandState& C, float* sv, int* si, float x, int i, int k) {
    const int lane = threadIdx.x & 31;
    unsigned m = __ballot_sync(FULL, C.wants(x));
    if (C.n + __popc(m) > kCandCap) {
        C = cand_compact<DT>(C, sv, si, k);
        m = __ballot_sync(FULL, C.wants(x));
    }
    if ((m >> lane) & 1u) {
        const int o = C.n + __popc(m & ((1u << lane) - 1u));
        sv[o] = x;
        si[o] = i;
    }
    C.n += __popc(m);
    __syncwarp();
}

// Next bf16 value below x (x a bf16 value, not NaN, not -inf): with it,
// "y >= x" is "y > bf16_pred(x)" for every bf16 y.
__device__ __forceinline__ uint32_t bf16_pred(uint32_t xb) {
    if (xb == 0x0000u || xb == 0x8000u) return 0x8001u;  // +-0 -> the negative denormal next to zero
    return (xb & 0x8000u) ? xb + 1u : xb - 1u;
}

// candidate bits of the 8 tokens of a bf16 vector: bit e iff token e > the
// bf16 pair tt (packed max, then compare with tt; NaN halves lose the max)
__device__ __forceinline__ uint32_t bf16_vec_bits(const uint4& d, uint32_t tt) {
    const uint32_t z0 = bf2_max(d.x, tt) ^ tt, z1 = bf2_max(d.y, tt) ^ tt;
    const uint32_t z2 = bf2_max(d.z, tt) ^ tt, z3 = bf2_max(d.w, tt) ^ tt;
    return (uint32_t)((z0 & 0xffffu) != 0) | ((uint32_t)((z0 >> 16) != 0) << 1) |
           ((uint32_t)((z1 & 0xffffu) != 0) << 2) | ((uint32_t)((z1 >> 16) != 0) << 3) |
           ((uint32_t)((z2 & 0xffffu) != 0) << 4) | ((uint32_t)((z2 >> 16) != 0) << 5) |
           ((uint32_t)((z3 & 0xffffu) != 0) << 6) | ((uint32_t)((z3 >> 16) != 0) << 7);
}

// Append the wanted tokens of this lane's flagged vectors (bit j of vf: the
// vector staged at st[j * 32 + lane]) to the buffer, compacting it when they
// do not fit (then the rest are re-tested against the raised threshold).
// Out of line: the scan keeps no token array in registers across it.
template <int DT>
__device__ __forceinline__ float staged_token(const uint4* st, int j, int e, int lane) {
    const uint4* vp = st + j * 32 + lane;
    if constexpr (DT == 1) return __uint_as_float((uint32_t)reinterpret_cast<const unsigned short*>(vp)[e] << 16);
    else return reinterpret_cast<const float*>(vp)[e];
}

template <int DT>
__device__ __noinline__ CandState cand_append(CandState C, float* sv, int* si, const uint4* st, unsigned vf,
                                              int i0, int k) {
    constexpr int VW = DT == 1 ? 8 : 4;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    while (true) {
        // candidate bits, VW per flagged vector
        uint64_t mask = 0;
        if constexpr (DT == 1) {
            // packed test against the pair tt (a superset: +-0 may tie), then the exact test per bit
            const bool strict = C.thr == -kInf || !(C.dropmax < C.thr);
            const uint32_t tb = __float_as_uint(C.thr) >> 16;
            const uint32_t t1 = strict ? tb : bf16_pred(tb);
            const uint32_t tt = t1 | (t1 << 16);
            for (unsigned m = vf; m; m &= m - 1) {
                const int j = __ffs(m) - 1;
                mask |= (uint64_t)bf16_vec_bits(st[j * 32 + lane], tt) << (j * VW);
            }
            for (uint64_t m = mask; m; m &= m - 1) {
                const int b = __ffsll((long long)m) - 1;
                if (!C.wants(staged_token<DT>(st, b / VW, b % VW, lane))) mask &= ~(1ull << b);
            }
        } else {
            for (unsigned m = vf; m; m &= m - 1) {
                const int j = __ffs(m) - 1;
                uint32_t b = 0;
#pragma unroll
                for (int e = 0; e < 4; ++e) b |= (uint32_t)C.wants(staged_token<DT>(st, j, e, lane)) << e;
                mask |= (uint64_t)b << (j * VW);
            }
        }
        const int cnt = __popcll(mask);
        int off = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL, off, o);
            if (lane >= o) off += t;
        }
        const int total = __shfl_sync(FULL, off, 31);
        off -= cnt;
        const bool fits = C.n + off + cnt <= kCandCap;
        if (fits) {
            int o = C.n + off;
            for (uint64_t m = mask; m; m &= m - 1) {
                const int b = __ffsll((long long)m) - 1, j = b / VW, e = b % VW;
                sv[o] = staged_token<DT>(st, j, e, lane);
                si[o] = i0 + 32 * VW * j + e;
                ++o;
            }
        }
        const unsigned done = __ballot_sync(FULL, fits);  // a prefix of the lanes
        if (done == FULL) {
            C.n += total;
            __syncwarp();
            return C;
        }
        const int last = 31 - __clz(done | 1u);
        C.n += done ? __shfl_sync(FULL, off + cnt, last) : 0;
        if (fits) vf = 0;
        __syncwarp();
        C = cand_compact<DT>(C, sv, si, k);
    }
}

// Flagged vectors wait in a per-warp queue of their indexes; one iteration adds
// at most 32 x NV.  Working the queue off loads the vectors again (they are in
// L2), 5 KB of shared memory less a CTA, which the L1 gets.
constexpr int kTQueueCap = 32 + 32 * PPS_TRUNC_UNITS;

// Work off the queue, one vector per lane (staged in st), 32 at a time.
template <int DT>
__device__ __noinline__ CandState topk_flush(CandState C, float* sv, int* si, uint4* st, const uint32_t* qi, int qn,
                                             const char* row, int h, int k) {
    constexpr int VW = DT == 1 ? 8 : 4;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    for (int base = 0; base < qn; base += 32) {
        const bool mine = base + lane < qn;
        const uint32_t v = mine ? qi[base + lane] : 0u;
        if (mine) st[lane] = __ldg(reinterpret_cast<const uint4*>(row) + v);
        C = cand_append<DT>(C, sv, si, st, mine ? 1u : 0u, (int)(v * VW) + h, k);
    }
    // raise the threshold early: a stale one lets through many more tokens
    if (C.n >= PPS_TRUNC_EAGER) C = cand_compact<DT>(C, sv, si, k);
    return C;
}

// One iteration of the fast scan (NV vectors per lane, d[j] = vector vfirst +
// 32 j; past the segment's end -inf, which no threshold lets through): a packed max tree per lane
// and a vote; vectors with a logit at or over the threshold are queued, and the queue is worked off
// once it holds 32.
template <int DT>
__device__ __forceinline__ void topk_step(CandState& C, float* sv, int* si, uint4* st, uint32_t* qi, int& qn,
                                          const uint4 (&d)[PPS_TRUNC_UNITS], const char* row, int64_t vfirst,
                                          int h, int k) {
    constexpr int NV = PPS_TRUNC_UNITS;
    const int lane = threadIdx.x & 31;
    // with no threshold yet (fewer than k usable tokens so far) a vector of nothing but -inf, a masked
    // stretch of the vocabulary, still has none to offer
    const float thr = fmaxf(C.thr, -FLT_MAX);
    unsigned vf = 0;
    if constexpr (DT == 1) {
        const uint32_t tb = __float_as_uint(thr) >> 16;  // a bf16 value on bf16 rows
        const uint32_t t2 = tb | (tb << 16);
        uint32_t mv[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) mv[j] = bf2_max(bf2_max(d[j].x, d[j].y), bf2_max(d[j].z, d[j].w));
        uint32_t m = mv[0];
#pragma unroll
        for (int j = 1; j < NV; ++j) m = bf2_max(m, mv[j]);
        const bool hit = bf2_any_ge(m, t2);
        if (!__any_sync(FULL, hit)) return;
        if (hit) {
#pragma unroll
            for (int j = 0; j < NV; ++j) vf |= (unsigned)bf2_any_ge(mv[j], t2) << j;
        }
    } else {
        float mv[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) mv[j] = vecs_max<DT>(d, j, 1);
        float m = mv[0];
#pragma unroll
        for (int j = 1; j < NV; ++j) m = fmaxf(m, mv[j]);
        const bool hit = m >= thr;
        if (!__any_sync(FULL, hit)) return;
        if (hit) {
#pragma unroll
            for (int j = 0; j < NV; ++j) vf |= (unsigned)(mv[j] >= thr) << j;
        }
    }
    const int n = __popc(vf);
    int off = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, off, o);
        if (lane >= o) off += t;
    }
    const int total = __shfl_sync(FULL, off, 31);
    off += qn - n;
    for (; vf; vf &= vf - 1) qi[off++] = (uint32_t)vfirst + 32u * (uint32_t)(__ffs(vf) - 1);
    qn += total;
    if (qn >= 32) {
        C = topk_flush<DT>(C, sv, si, st, qi, qn, row, h, k);
        qn = 0;
    }
}

// The fast scan of vectors [v0, vend) of a row's aligned interior (`row`: its
// start, token h of the row): iterations of NV vectors 32 apart per lane; in
// the last, partial one the vectors past vend read as -inf.  The first
// iteration also seeds the threshold.
template <int DT>
__device__ __forceinline__ void topk_scan(CandState& C, float* sv, int* si, uint4* st, uint32_t* qi,
                                          const char* row, int64_t v0, int64_t vend, int h, int k, float guess) {
    constexpr int NV = PPS_TRUNC_UNITS;
    constexpr int STEP = 32 * NV;
    const int lane = threadIdx.x & 31;
    const uint32_t ninf = DT == 1 ? 0xff80ff80u : 0xff800000u;
    const uint4 fill = make_uint4(ninf, ninf, ninf, ninf);
    const int64_t n_it = (vend - v0 + STEP - 1) / STEP;
    const uint4* p = reinterpret_cast<const uint4*>(row) + v0 + lane;
    int qn = 0;
    for (int64_t it = 0; it < n_it; ++it) {
        const int64_t vb = v0 + it * STEP + lane;
        uint4 d[NV];
        if (v0 + (it + 1) * STEP <= vend) {
#pragma unroll
            for (int j = 0; j < NV; ++j) d[j] = ldg_stream(p + 32 * j);
        } else {
#pragma unroll
            for (int j = 0; j < NV; ++j) d[j] = vb + 32 * j < vend ? ldg_stream(p + 32 * j) : fill;
        }
        p += STEP;
        if (it == 0) C.thr = fmaxf(guess, seed_thr<DT>(d, k));
        topk_step<DT>(C, sv, si, st, qi, qn, d, row, vb, h, k);
    }
    if (qn > 0) C = topk_flush<DT>(C, sv, si, st, qi, qn, row, h, k);
}

// Segment [v0, v1) (in units of the row partition) of a row.  Finding S needs no
// Philox words, so vectors need not line up with blocks: the scan takes the
// row's aligned interior, nfull vectors from its first 16-byte boundary on (h
// tokens in), and the at most 2 (VW - 1) tokens before and after it are
// offered one per lane, by the segments that hold the row's start and end.
// Rows of any alignment stream at the same rate: 16720 rows of V = 5717 bf16,
// top-k 50, took 736 us when unaligned rows were read one token at a time, 382 with
// this change alone.
template <int DT>
__device__ __forceinline__ CandState topk_segment(const char* row, int64_t V, int64_t v0, int64_t v1, int64_t nv, int k,
                                                  float* sv, int* si, uint4* st, uint32_t* qi) {
    constexpr int VW = DT == 1 ? 8 : 4;
    constexpr int ESZ = DT == 1 ? 2 : 4;
    const int lane = threadIdx.x & 31;
    const int h = (int)min(V, (int64_t)((0u - (uint32_t)reinterpret_cast<uintptr_t>(row)) & 15u) / ESZ);
    const int64_t nfull = (V - h) / VW;
    const int64_t vend = min(v1, nfull);
    CandState C{-kInf, -kInf, 0};
    if (vend > v0) {
        const char* in = row + h * ESZ;
        float guess = vend - v0 >= kSampleMin ? guess_thr<DT>(in, v0, vend, k) : -kInf;
        while (true) {
            topk_scan<DT>(C, sv, si, st, qi, in, v0, vend, h, k, guess);
            if (C.n >= k || guess == -kInf) break;
            guess = -kInf;  // fewer than k tokens reached the guess: scan again from the proven threshold alone
            C = CandState{-kInf, -kInf, 0};
        }
    }
    const int64_t t0 = h + nfull * VW;  // the tokens after the interior
    const int nh = v0 == 0 ? h : 0, nt = v1 == nv ? (int)(V - t0) : 0;
    if (nh + nt > 0) {
        const int64_t i = lane < 16 ? lane : t0 + (lane - 16);
        float x = -kInf;
        if (lane < 16 ? lane < nh : lane - 16 < nt) x = load_logit<DT>(row, i);
        cand_push<DT>(C, sv, si, x, (int)i, k);
    }
    return C;
}

// ---------------------------------------------------------------- finishing a truncated row

template <int DT>
__device__ __noinline__ int64_t count_logit(const char* row, int64_t V, float x) {
    const int lane = threadIdx.x & 31;
    long long n = 0;
    for (int64_t i = lane; i < V; i += 32) n += load_logit<DT>(row, i) == x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(FULL, n, o);
    return (int64_t)n;
}

// Top-p on the kept-by-top-k set: the list's entries with logit >= lk (a
// prefix, in top order) plus `extra` more tokens of logit lk that the list
// could not hold.  The lanes form the exponentials and the probabilities; lane 0
// adds them in ascending order, exactly as the definition sums, and walks the
// groups; returns the smallest kept logit (every token >= it stays).  (All of
// it on one lane: 11 sequences, V = 7338, top-k 16, top-p 0.9, 111 us a step
// instead of 65.)
__device__ __noinline__ float top_p_keep(const TopList& L, float lk, int64_t extra, float top_p, float T,
                                         float* s_val, double* s_e) {
    const int lane = threadIdx.x & 31;
    const bool ka = L.av > -kInf && L.av >= lk, kb = L.bv > -kInf && L.bv >= lk;
    const int nk = __popc(__ballot_sync(FULL, ka)) + __popc(__ballot_sync(FULL, kb));
    const double top = (double)__shfl_sync(FULL, L.av, 0), Td = (double)T, cut = 1.0 - (double)top_p;
    const double ex = exp(((double)lk - top) / Td);
    const double ea = ka ? exp(((double)L.av - top) / Td) : 0.0, eb = kb ? exp(((double)L.bv - top) / Td) : 0.0;
    s_val[lane] = L.av;
    s_val[32 + lane] = L.bv;
    s_e[lane] = ea;
    s_e[32 + lane] = eb;
    __syncwarp();
    double Z = 0.0;  // every lane sums alike
    for (int64_t t = 0; t < extra; ++t) Z += ex;
    for (int j = nk - 1; j >= 0; --j) Z += s_e[j];
    __syncwarp();
    s_e[lane] = ea / Z;
    s_e[32 + lane] = eb / Z;
    __syncwarp();
    const double px = ex / Z;
    double run = 0.0;
    for (int64_t t = 0; t < extra; ++t) run += px;
    float keep = s_val[0];
    for (int j = nk - 1; j >= 0; --j) {
        run += s_e[j];
        if (j > 0 && s_val[j - 1] == s_val[j]) continue;  // not the end of its group
        if ((double)s_val[j] == top) break;               // the top group stays
        if (run <= cut) {
            keep = s_val[j - 1];
        } else {
            keep = s_val[j];
            break;
        }
    }
    __syncwarp();
    return keep;
}

// lower 32 of two lists sorted ascending by (key, token): into x; returns the lane's key of the upper 32
__device__ __forceinline__ float merge_low_f(float& xk, int& xi, float yk, int yi, int lane) {
    const float rk = __shfl_sync(FULL, yk, 31 - lane);
    const int ri = __shfl_sync(FULL, yi, 31 - lane);
    float up = rk;
    if (lex_less(rk, ri, xk, xi)) {
        up = xk;
        xk = rk;
        xi = ri;
    }
#pragma unroll
    for (int stride = 16; stride > 0; stride >>= 1) {
        const float ok = __shfl_xor_sync(FULL, xk, stride);
        const int oi = __shfl_xor_sync(FULL, xi, stride);
        const bool lower = (lane & stride) == 0;
        const bool o_less = lex_less(ok, oi, xk, xi);
        if (lower ? o_less : (!o_less && !(ok == xk && oi == xi))) {
            xk = ok;
            xi = oi;
        }
    }
    return up;
}

// Finish a row when more keys crowd its K-th, tau, than the kept list holds: the
// K smallest of S (the n buffered tokens with logit >= keep) by their fp64 keys.
// About one row of K = 32 in 4000 comes here; sorting (three rolled sorts) instead of picking
// the smallest 32 times, and the fp32 epilogue of IID rows, which tests every gap that decides a
// sample, keep a launch from waiting for it (4096 rows of V = 1000 fp32: 82 -> 78 us, 76.5 with none of this).
template <int DT, bool VERIFY, bool BLK>
__device__ __noinline__ void finish_crowded(const RaceArgs& a, int64_t r, float tau, int n, float keep, int kr,
                                            const float* sv, const int* si, Blk bk) {
    const int lane = threadIdx.x & 31;
    const uint64_t key = a.key[r], ctx = a.ctx[r];
    const uint32_t pos = a.pos[r];
    if (lane == 0 && a.status && fabsf(tau) > 65536.0f) atomicOr(a.status, PPS_FLAG_LOGIT_RANGE);
    double d[2];
    int id[2], size = 0;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int m = 32 * t + lane;
        const float l = m < n ? sv[m] : -kInf;
        const bool in = l > -kInf && l >= keep;
        id[t] = in ? si[m] : INT_MAX;
        d[t] = in ? exact_key<BLK>(key, ctx, pos, id[t], l, a.T, bk) : (double)INFINITY;
        size += __popc(__ballot_sync(FULL, in));
    }
    // the lower 32 of both halves, in order
    warp_sort_d(d[0], id[0], lane);
    warp_sort_d(d[1], id[1], lane);
    const double rd = __shfl_sync(FULL, d[1], 31 - lane);
    const int ri = __shfl_sync(FULL, id[1], 31 - lane);
    if (lex_less_d(rd, ri, d[0], id[0])) {
        d[0] = rd;
        id[0] = ri;
    }
    warp_sort_d(d[0], id[0], lane);
    const int nvalid = min(size, 32);
    const auto logits = dense_logits<DT>(a, r);
    if constexpr (!VERIFY && !BLK) {
        if (a.iid && PPS_IID_FAST) {
            const float lk = lane < nvalid ? key32(word_of(key, ctx, pos, id[0], 1), logits(id[0]), a.c) : kInf;
            if (iid_fast<DT>(a, r, lk, id[0], nvalid, kr, lane, key, ctx, pos, logits)) return;
        }
    }
    emit_row<DT, VERIFY>(a, r, d[0], (float)d[0], id[0], nvalid, kr, lane, key, ctx, pos, logits);
}

// Finish row r from its buffer, which holds every token at or over l_(k) but
// those dropmax tells of.  S comes straight from the buffer: one more
// compaction leaves the tokens >= l_(k); nothing is sorted but the race keys
// (short lists by kp rounds of a warp argmin, others by a warp sort).
template <int DT, bool VERIFY, bool BLK>
__device__ __noinline__ void finalize_trunc(const RaceArgs& a, int64_t r, CandState C, int kr, int kp, float* sv,
                                            int* si, float* s_val, double* s_e, Blk bk) {
    const int lane = threadIdx.x & 31;
    const int k = a.top_k;
    float lk = -kInf;  // l_(k); -inf when the row has fewer than k usable tokens
    if (C.n >= k) {
        C = cand_compact<DT>(C, sv, si, k);
        lk = C.thr;
    }
    const bool over = lk > -kInf && C.dropmax >= lk;
    const char* row = reinterpret_cast<const char*>(a.logits) + (size_t)r * (size_t)a.stride * (DT == 1 ? 2 : 4);
    const uint64_t key = a.key[r], ctx = a.ctx[r];
    const uint32_t pos = a.pos[r];
    float keep = lk;
    if (a.top_p < 1.0f) {
        const TopList L = cand_to_list(C.n, sv, si);
        int64_t extra = 0;
        if (over) {
            const int in_list = __popc(__ballot_sync(FULL, L.av == lk)) + __popc(__ballot_sync(FULL, L.bv == lk));
            extra = count_logit<DT>(row, a.V, lk) - in_list;
        }
        keep = top_p_keep(L, lk, extra, a.top_p, a.T, s_val, s_e);
    }
    if (over && keep <= lk) {
        // the tie group of l_(k) stays but is not all in the list: exact race
        // over every token with logit >= l_(k), one pass of the scalar path
        WarpList W;
        W.reset(kp, kr);
        SlowState st{W};
        st = tail_loop<DT, BLK>(st, row, a.V, 0, a.nv, a.c, key, ctx, pos, lk, bk, reinterpret_cast<uint64_t*>(sv));
        finalize_row<DT, VERIFY, BLK>(a, r, st.L.lk, st.L.li, st.L.drop(), kr, kp, lane, bk,
                                      reinterpret_cast<uint32_t*>(si), lk);
        return;
    }
    // S = the buffer's entries with logit >= keep: the race's fp32 keys, the kp
    // smallest in lane order, and `left`, the smallest key of the others.  When it
    // is beyond the K-th key's error bounds, finalize_row re-keys near ties in fp64
    float kk[2];
    int ii[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int m = 32 * t + lane;
        const float l = m < C.n ? sv[m] : -kInf;
        kk[t] = kInf;
        ii[t] = m < C.n ? si[m] : INT_MAX;
        if (l > -kInf && l >= keep) {
            const uint32_t w = word_of(key, ctx, pos, ii[t], 1);
            // proposal rows of the augmented race: the tokens' block arrivals
            if constexpr (BLK) kk[t] = block_key_of(key, ctx, pos, ii[t], w, l, a.c, bk.b, bk.B, bk.invB());
            else kk[t] = key32(w, l, a.c);
        }
        if (kk[t] == kInf) ii[t] = INT_MAX;
    }
    float ka = kInf, left;
    int ia = INT_MAX;
    if (kp <= kTruncRounds) {
        for (int m = 0; m < kp; ++m) {
            const bool second = lex_less(kk[1], ii[1], kk[0], ii[0]);
            float bk_;
            const int bi = warp_argmin(second ? kk[1] : kk[0], second ? ii[1] : ii[0], bk_);
            if (bi == INT_MAX) break;
            if (lane == m) {
                ka = bk_;
                ia = bi;
            }
#pragma unroll
            for (int t = 0; t < 2; ++t)
                if (ii[t] == bi) {
                    kk[t] = kInf;
                    ii[t] = INT_MAX;
                }
        }
        left = fminf(kk[0], kk[1]);
    } else {
        warp_sort(kk[0], ii[0], lane);
        warp_sort(kk[1], ii[1], lane);
        left = merge_low_f(kk[0], ii[0], kk[1], ii[1], lane);
        ka = kk[0];
        ia = ii[0];
        if (lane >= kp) left = fminf(left, ka);
    }
    left = warp_min(left);
    const float tau = __shfl_sync(FULL, ka, kr - 1), eb = BLK ? kBlkErr : 0.f;
    if (left < kInf && tau > -kInf && !(left > tau + key_err_bound(tau) + key_err_bound(left) + 2.0f * eb)) {
        finish_crowded<DT, VERIFY, BLK>(a, r, tau, C.n, keep, kr, sv, si, bk);
        return;
    }
    finalize_row<DT, VERIFY, BLK>(a, r, ka, ia, kInf, kr, kp, lane, bk);
}

// End of a row segment: publish the segment's buffer (its at most 64 largest
// tokens), or finish the row if the warp is the last of the row to arrive.  Each
// segment's threshold bounds l_(k) from below, so of all published tokens only those
// at or over the largest threshold are gathered again: about as many as one
// segment holds, whatever their number.  (Merging the sorted lists of 74
// segments one after another took most of the 263 us of a one-sequence step.)
template <int DT, bool VERIFY, bool BLK>
__device__ __noinline__ void finish_trunc_segment(const RaceArgs& a, int64_t r, int64_t gw, int64_t NW, int64_t v0,
                                                  int64_t v1, CandState C, int kr, int kp, float* sv, int* si,
                                                  float* s_val, double* s_e, Blk bk) {
    const int lane = threadIdx.x & 31;
    const int64_t nv = a.nv;
    const int k = a.top_k;
    bool final_here = v0 == 0 && v1 == nv;
    if (!final_here) {
        if (C.n >= k) C = cand_compact<DT>(C, sv, si, k);
        TruncPartial* P = a.tpartials + (gw + r);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int m = 32 * t + lane;
            P->v[m] = m < C.n ? sv[m] : -kInf;
            P->idx[m] = m < C.n ? si[m] : INT_MAX;
        }
        if (lane == 0) {
            P->dropmax = C.dropmax;
            P->thr = C.thr;
        }
        __threadfence();
        __syncwarp();
        const int64_t first_w = warp_of(r * nv, a.total, NW);
        const int64_t last_w = warp_of(r * nv + nv - 1, a.total, NW);
        unsigned last = 0;
        if (lane == 0) {
            unsigned t = atomicAdd(a.row_cnt + r, 1u);
            last = t == (unsigned)(last_w - first_w);
            if (last) a.row_cnt[r] = 0u;
        }
        final_here = __shfl_sync(FULL, last, 0) != 0;
        if (final_here) {
            __threadfence();
            float thr = -kInf, dropmax = -kInf;
            for (int64_t ww = first_w + lane; ww <= last_w; ww += 32) {
                thr = fmaxf(thr, __ldcg(&a.tpartials[ww + r].thr));
                dropmax = fmaxf(dropmax, __ldcg(&a.tpartials[ww + r].dropmax));
            }
            C.thr = from_order_key(__reduce_max_sync(FULL, order_key(thr)));
            dropmax = from_order_key(__reduce_max_sync(FULL, order_key(dropmax)));
            C.dropmax = -kInf;  // gathers the ties of the threshold that were kept
            C.n = 0;
            for (int64_t ww = first_w; ww <= last_w; ww += 4) {
                float v[8];
                int ix[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const bool on = ww + (j >> 1) <= last_w;
                    const TruncPartial* Q = a.tpartials + (ww + (j >> 1) + r);
                    v[j] = on ? __ldcg(Q->v + 32 * (j & 1) + lane) : -kInf;
                    ix[j] = on ? __ldcg(Q->idx + 32 * (j & 1) + lane) : INT_MAX;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) cand_push<DT>(C, sv, si, v[j], ix[j], k);
            }
            C.dropmax = fmaxf(C.dropmax, dropmax);
        }
    }
    if (final_here) {
        finalize_trunc<DT, VERIFY, BLK>(a, r, C, kr, kp, sv, si, s_val, s_e, bk);
        if constexpr (VERIFY) sequence_ticket(a, r, lane);
    }
}

// ---------------------------------------------------------------- the kernel

template <int DT, bool VERIFY, bool BLK>
__global__ void __launch_bounds__(kThreads, PPS_TRUNC_MIN_BLOCKS) trunc_kernel(const RaceArgs a) {
    __shared__ __align__(16) float s_cv[kCandCap];
    __shared__ int s_ci[kCandCap];
    __shared__ uint4 s_st[32];
    __shared__ __align__(16) uint32_t s_qi[kTQueueCap];
    // top-p works on the finished row, when the queue is empty
    double* s_e = reinterpret_cast<double*>(s_qi);
    float* s_val = reinterpret_cast<float*>(s_e + kTopMax);
    static_assert(sizeof(s_qi) >= kTopMax * (sizeof(double) + sizeof(float)), "top-p's exponentials and logits");
    pdl_wait();  // the previous kernel's outputs and the workspace it used
    pdl_launch_dependents();
    const int64_t NW = a.G;
    const int64_t gw = blockIdx.x;
    const int64_t g0 = gw * a.total / NW, g1 = (gw + 1) * a.total / NW;
    const int64_t nv = a.nv;
    const size_t esz = DT == 1 ? 2 : 4;

    for (int64_t r = g0 / nv; g0 < g1 && r < a.n_rows && r * nv < g1; ++r) {
        const int64_t v0 = max(g0, r * nv) - r * nv, v1 = min(g1, (r + 1) * nv) - r * nv;
        int kr = 1;
        if (!VERIFY) {
            kr = a.row_k ? __ldg(a.row_k + r) : a.K;
            kr = max(1, min(kr, a.K));
        }
        const int kp = min(32, 2 * kr + 1);
        const char* row = reinterpret_cast<const char*>(a.logits) + (size_t)r * (size_t)a.stride * esz;
        const CandState C = topk_segment<DT>(row, a.V, v0, v1, nv, a.top_k, s_cv, s_ci, s_st, s_qi);
        Blk bk;
        if constexpr (BLK) {
            bk.b = __ldg(a.row_block + r);
            bk.B = a.n_blocks;
        }
        finish_trunc_segment<DT, VERIFY, BLK>(a, r, gw, NW, v0, v1, C, kr, kp, s_cv, s_ci, s_val, s_e, bk);
    }
}
