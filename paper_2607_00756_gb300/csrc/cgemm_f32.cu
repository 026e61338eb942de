// FP32 complex contractions on the tensor cores (tcgen05), operands cut into
// three BF16 terms inside the kernel.
//
//   coupling   M^{(n)}_{d,b} = sum_r S2^d(r) [H_n S1^b](r)          (Eq. coupling)
//   Gram       Q_{b,b'} = sum_{n,d} conj(M^{(n)}_{d,b}) M^{(n)}_{d,b'}
// (the exact regrouping of Eq. map-sum: sum_n sum_d |sum_b M_{d,b} c_b|^2 =
// c^H Q c; c^H Q c itself is evaluated in difftrans.cu), and the
// contractions of the reverse pass (grad.cu states them).
//
// C(m, n) = sum_k opA(A(m, k) w_k) opB(B(k, n)), complex64 in and out.
// x = x0 + x1 + x2 with x0 = bf16(x), x1 = bf16(x - x0), x2 = bf16(x - x0 - x1)
// keeps 24 bits of every element; of the nine products of a real product the
// six down to 2^-18 of the leading one are taken (the dropped ones are below
// 2^-26).  Accuracy of the sums: a chunk of 16 complex k is summed in TMEM,
// the five small products first and the leading one last, so only two MMAs add
// at full magnitude per chunk; the chunks are then added in FP32 registers with
// round-to-nearest.  That is 16x fewer roundings per sum than a fused
// multiply-add per k, and no long run of tensor-core additions.  The whole FP32
// range is taken, infinities and NaN as such; elements below 2^-110 (7.7e-34)
// lose the last of their 24 bits, as BF16 ends at 2^-133.
//
// The complex product as one real one: an A row holds [Re (16) | Im (16)] of a
// chunk (64 bytes), B has two rows per column n, [Re | -Im] for the real part
// of C and [Im | Re] for the imaginary part, so that one MMA of N = 2 nt covers
// both parts: 12 MMAs (M = 128, N <= 256, K = 16) per chunk.
//
// Persistent, one CTA per SM, 20 warps in five warpgroups, which divide the
// registers anew at the start (setmaxnreg):
//   warps 0-7    load the elements of the next chunk (FP32, from L2) into
//                registers and cut the present ones into the three terms in
//                a 3-stage shared ring (64 registers);
//   warps 8-15   add finished chunks from TMEM (two accumulator sets) to their
//                sums: warp w owns TMEM lanes 32 (w % 4) .. and 64 columns of
//                the tile, Re and Im, in 128 registers (of 152);
//   warp 16      TMEM allocator and MMA issuer (40; warps 17-19 idle).
// What bounds it: the cutting warps (latency: the loads of a chunk, then about
// 500 dependent instructions per warp), 2800 clocks per chunk of a 128 x 128
// tile where its twelve MMAs take about 1900.  Measured on 19 x 1024 x 1024 x 4096:
// 220 TFLOP/s of complex products (SIMT FFMA, 64 x 64 tiles: 47); two groups
// of four cutting warps taking chunks in turn 209-218, sixteen cutting warps
// of 40 registers 160, loads issued between the cutting of A and of B 219, two
// CTAs sharing a tile of 256 rows (cta_group::2, each with half of B) 192-212.
//
// Units: (batch, tile of 128 rows, tile of nt columns, k range).  Where the
// tiles alone leave SMs idle the k range is split (cgemm_plan), each part
// written to a workspace and added in order by cgemm_sum_kernel: the result
// does not depend on scheduling.  Every wait is bounded; on a timeout the
// kernel sets *err, stops issuing, drains its MMAs and frees TMEM.
#include <algorithm>

#include "tc_common.cuh"

namespace {

constexpr int kCut = 8, kAdd = 8;                // warps that cut, warps that add
constexpr int kIssuer = kCut + kAdd;
constexpr int kThreads = 32 * (kIssuer + 4);
constexpr int kRegsLaunch = 96, kRegsCut = 64, kRegsAdd = 152, kRegsIssue = 40;
static_assert(32 * (kCut * kRegsCut + kAdd * kRegsAdd + 4 * kRegsIssue) <= kThreads * kRegsLaunch,
              "the split draws on the registers of the launch");
static_assert(kRegsCut <= kRegsLaunch && kRegsIssue <= kRegsLaunch && kRegsAdd >= kRegsLaunch,
              "setmaxnreg.dec gives registers back, .inc takes some");
constexpr int kStep = 16;                        // complex k per chunk
constexpr int kALevel = 128 * 64, kBLevel = 256 * 64;   // bytes of one term of a stage
constexpr int kStage = 3 * (kALevel + kBLevel);
constexpr int kStages = 3;
constexpr size_t kSmem = 1024 + (size_t)kStages * kStage + 256;

// mbar_wait of tc_common.cuh whose tries sleep up to 2 us each: twenty warps
// wait here most of the time, and their polling took issue slots from the
// cutting
__device__ __forceinline__ bool mbar_try_long(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity), "r"(2000u)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool wait_long(uint64_t* b, uint32_t parity, volatile int* abort_flag, uint64_t limit) {
    if (limit < 1000000ull) return mbar_wait(b, parity, abort_flag, limit);
    if (mbar_try_long(b, parity)) return true;
    const uint64_t t0 = gtimer();
    for (;;) {
        if (mbar_try_long(b, parity)) return true;
        if (*abort_flag || gtimer() - t0 > limit) return false;
    }
}

struct Unit {
    int z, m0, n0, n1, ks;                       // columns [n0, n1)
    int s0, s1;                                  // steps [s0, s1)
};

__device__ __forceinline__ bool unit_of(const CGemmF32& p, int i, Unit& u) {
    int idx = blockIdx.x + i * gridDim.x;
    if (idx >= p.units) return false;
    u.ks = idx % p.ksplit;
    idx /= p.ksplit;
    u.z = idx / p.tiles;
    int r = idx % p.tiles;
    if (p.tri) {
        // row tile mt keeps the column tiles from mt 128 / nt on
        int mt = 0;
        for (;; ++mt) {
            const int first = mt * 128 / p.nt;
            const int n = p.n_tiles - first;
            if (r < n) {
                r += first;
                break;
            }
            r -= n;
        }
        u.m0 = mt * 128;
    } else {
        u.m0 = r / p.n_tiles * 128;
        r %= p.n_tiles;
    }
    u.n0 = r * p.nt;
    u.n1 = min(u.n0 + p.nt, p.cols);
    u.s0 = (int)((int64_t)p.steps * u.ks / p.ksplit);
    u.s1 = (int)((int64_t)p.steps * (u.ks + 1) / p.ksplit);
    return true;
}

// One chunk of an operand (128 rows x 16 k) over the eight cutting warps, 16
// rows per warp.  KC (k contiguous): eight lanes take the 16 k of a row, two
// each, four rows {0, 1, 4, 5} + {0, 2, 8, 10} of the warp's at a time (with the
// 64-byte swizzle the 4-byte stores of such four rows hit every bank once).
// Else (rows contiguous): a thread takes four k of one row, twice.
template <bool KC>
struct Slot {
    int row, k;                                  // first row, first k within the chunk
    __device__ Slot(int warp, int lane) {
        if (KC) {
            const int g = lane >> 3;
            row = warp * 16 + (g & 1) + (g >> 1) * 4;
            k = 2 * (lane & 7);
        } else {
            row = warp * 16 + (lane >> 4) * 8 + (lane & 7);
            k = ((lane >> 3) & 1) * 4;
        }
    }
    // row and k of value i (of 8)
    __device__ int row_of(int i) const { return KC ? row + 2 * ((i >> 1) & 1) + 8 * (i >> 2) : row; }
    __device__ int k_of(int i) const { return KC ? k + (i & 1) : k + 8 * (i >> 2) + (i & 3); }
};

// row of B that column n of C comes from
__device__ __forceinline__ int row_of_column(const CGemmF32& p, int n) {
    return p.ep_B > 0 ? n / p.ep_n * p.ep_B + n % p.ep_n : n;
}

// the thread's eight values of chunk `step`, of its rows row[] (zeros past the
// last k).  Rows past the last were clamped to it: what they give reaches only
// rows and columns of C that are not written.
template <bool KC>
__device__ __forceinline__ void load8(float2 (&v)[8], const CGemmOperand& o, const float2* base,
                                      const int (&row)[KC ? 4 : 1], const Slot<KC>& sl, int step) {
    // block kb of the two-level k axis
    const int k0 = step * kStep;
    const int kb = o.nper > 1 ? k0 / o.kper : 0;
    const int kin = k0 - kb * o.kper;
    const float2* src = base + (int64_t)kb * o.sk2 + (KC ? kin + sl.k : (int64_t)(kin + sl.k) * (int)o.sk);
    const float2* at[KC ? 4 : 1];
#pragma unroll
    for (int i = 0; i < (KC ? 4 : 1); ++i) at[i] = src + (KC ? (int64_t)row[i] * (int)o.sr : row[i]);
    if (kin + kStep <= o.kvalid) {
        if (KC && o.vec) {
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const float4 f = __ldg(reinterpret_cast<const float4*>(at[KC ? i / 2 : 0]));
                v[i] = make_float2(f.x, f.y);
                v[i + 1] = make_float2(f.z, f.w);
            }
        } else if (KC) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __ldg(at[KC ? i / 2 : 0] + (i & 1));
        } else {
            const float2* q = at[0];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __ldg(q + ((i >> 2) * 8 + (i & 3)) * (int)o.sk);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v[i] = make_float2(0.f, 0.f);
            if (kin + sl.k_of(i) < o.kvalid)
                v[i] = __ldg(KC ? at[KC ? i / 2 : 0] + (i & 1) : at[0] + ((i >> 2) * 8 + (i & 3)) * (int)o.sk);
        }
    }
}

// two FP32 values as three BF16 pairs.  The first two terms stay finite: past
// the largest BF16 (3.3895e38) they are that, which leaves the rest to the
// last term, so the largest FP32 values are exact too and an infinite one
// comes out infinite in the last term.
__device__ __forceinline__ uint32_t rest(float& a, float& b) {
    uint32_t t;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(t) : "f"(b), "f"(a));
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\tsub.rn.f32x2 x, x, y;\n\t"
        "mov.b64 {%0, %1}, x;\n\t}"
        : "+f"(a), "+f"(b)
        : "f"(bf16_lo(t)), "f"(bf16_hi(t)));
    return t;
}
__device__ __forceinline__ void cut(float a, float b, uint32_t (&t)[3]) {
    t[0] = rest(a, b);
    t[1] = rest(a, b);
    t[2] = pack_bf16x2(a, b);
}

__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, uint32_t v, uint32_t w) {
    asm volatile("st.shared.v2.b32 [%0], {%1,%2};" ::"r"(a), "r"(v), "r"(w) : "memory");
}

// byte of (row, k) in a term's tile (64-byte rows, 64-byte swizzle), Re half;
// the Im half is at the same byte ^ 32, row + 8 at byte + 512
__device__ __forceinline__ uint32_t tile_byte(int row, int k) {
    return (uint32_t)(row * 64 + ((((k >> 3) ^ (row >> 1)) & 3) << 4) + (k & 7) * 2);
}

// the thread's values as three terms each into a stage; byte[i]: tile_byte of
// value 2 i's (k contiguous) or 4 i's row and k
template <bool KC, bool IS_B>
__device__ __forceinline__ void store8(const float2 (&v)[8], uint32_t stage, const uint32_t (&byte)[2],
                                       const Slot<KC>& sl, int nt) {
    constexpr uint32_t LEVEL = IS_B ? kBLevel : kALevel;
    const uint32_t base = stage + (IS_B ? 3 * kALevel : 0);
    const uint32_t im_rows = (uint32_t)nt * 64;  // B: the rows of C's imaginary part
    if (KC) {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            if (IS_B && sl.row_of(i) >= nt) continue;
            uint32_t re[3], im[3];
            cut(v[i].x, v[i + 1].x, re);
            cut(v[i].y, v[i + 1].y, im);
            const uint32_t a = base + byte[(i >> 1) & 1], b = a ^ 32;
            const uint32_t at = (i >> 2) * 512;
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                sts32(a + at + l * LEVEL, re[l]);
                sts32(b + at + l * LEVEL, IS_B ? im[l] ^ 0x80008000u : im[l]);
                if (IS_B) {
                    sts32(a + im_rows + at + l * LEVEL, im[l]);
                    sts32(b + im_rows + at + l * LEVEL, re[l]);
                }
            }
        }
    } else {
        if (IS_B && sl.row >= nt) return;
#pragma unroll
        for (int i = 0; i < 8; i += 4) {
            uint32_t r0[3], r1[3], i0[3], i1[3];
            cut(v[i].x, v[i + 1].x, r0);
            cut(v[i + 2].x, v[i + 3].x, r1);
            cut(v[i].y, v[i + 1].y, i0);
            cut(v[i + 2].y, v[i + 3].y, i1);
            const uint32_t a = base + byte[i >> 2], b = a ^ 32;
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                sts64(a + l * LEVEL, r0[l], r1[l]);
                if (IS_B) {
                    sts64(b + l * LEVEL, i0[l] ^ 0x80008000u, i1[l] ^ 0x80008000u);
                    sts64(a + im_rows + l * LEVEL, i0[l], i1[l]);
                    sts64(b + im_rows + l * LEVEL, r0[l], r1[l]);
                } else {
                    sts64(b + l * LEVEL, i0[l], i1[l]);
                }
            }
        }
    }
}

// acc += sixteen TMEM columns of this thread's lane, two columns per add.  The
// adds are volatile so that they stay behind their own load: gathered behind
// all of a chunk's loads they would need another 128 registers.
__device__ __forceinline__ void add16(uint64_t (&acc)[8], uint32_t taddr) {
    float v[16];
    tmem_ld16(taddr, v);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 8; ++j)
        asm volatile("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tadd.rn.f32x2 %0, %0, t;\n\t}"
                     : "+l"(acc[j])
                     : "f"(v[2 * j]), "f"(v[2 * j + 1]));
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}

// where C(m, n) of batch z lies
__device__ __forceinline__ int64_t out_at(const CGemmF32& p, int z, int m, int n) {
    int64_t o = (int64_t)z * p.scb;
    if (p.ep_B > 0)                              // the coupling as the Gram operand: n = (ch, b), m = d
        return o + (int64_t)(n % p.ep_n) * p.scn + (int64_t)(n / p.ep_n) * p.ep_Dp + m;
    return o + (int64_t)m * p.scm + (int64_t)n * p.scn;
}

template <bool AKC, bool BKC>
__global__ void __launch_bounds__(kThreads, 1) cgemm_f32_kernel(const __grid_constant__ CGemmF32 p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + kStages * kStage);
    uint64_t* empty = full + kStages;
    uint64_t* acc_full = empty + kStages;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* drain = acc_empty + 2;
    uint32_t* tmem_slot = (uint32_t*)(drain + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&full[i], kCut);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], kAdd);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kIssuer) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tmem_slot;

    auto fail = [&]() {
        *abort_flag = 1;
        *(volatile int*)p.err = 1;               // device memory, or pinned host memory
    };

    // lane 0 waits for its warp
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        int w = 1;
        if (lane == 0) {
            w = wait_long(bar, parity, abort_flag, wait_limit(p.wait_ns)) ? 1 : 0;
            if (!w) fail();
        }
        return __shfl_sync(0xffffffffu, w, 0) != 0;
    };

    if (warp >= kIssuer) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
        if (warp == kIssuer && lane == 0) {
            // ---------------- MMA issuer
            const uint32_t id = idesc(128, 2 * p.nt, false);
            int s = 0, a = 0;
            uint32_t ph = 0, aph = 0;
            bool any = false, ok = true;
            Unit u;
            for (int i = 0; ok && unit_of(p, i, u); ++i) {
                for (int st = u.s0; st < u.s1; ++st) {
                    if (!wait_long(&acc_empty[a], aph ^ 1, abort_flag, wait_limit(p.wait_ns)) ||
                        !wait_long(&full[s], ph, abort_flag, wait_limit(p.wait_ns))) {
                        fail();
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(smem + s * kStage), sb = sa + 3 * kALevel;
                    const uint32_t d = tbase + (uint32_t)(a * 256);
                    // the small products first, the leading one last
                    constexpr int la[6] = {0, 2, 1, 0, 1, 0}, lb[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
                    for (int t = 0; t < 6; ++t)
#pragma unroll
                        for (int h = 0; h < 2; ++h)   // Re, then Im of A
                            mma(d, sdesc(sa + la[t] * kALevel + h * 32), sdesc(sb + lb[t] * kBLevel + h * 32), id,
                                t + h > 0 ? 1u : 0u);
                    any = true;
                    mma_commit(&empty[s]);
                    mma_commit(&acc_full[a]);
                    if (++s == kStages) {
                        s = 0;
                        ph ^= 1;
                    }
                    if (++a == 2) {
                        a = 0;
                        aph ^= 1;
                    }
                }
            }
            if (any) {
                mma_commit(drain);
                const uint64_t t0 = gtimer();
                while (!mbar_try(drain, 0) && gtimer() - t0 < kTimeoutNs) {
                }
            }
        }
    } else if (warp < kCut) {
        // ---------------- cut the operands into the ring
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsCut));
        const Slot<AKC> sla(warp, lane);
        const Slot<BKC> slb(warp, lane);
        uint32_t byteA[2], byteB[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            byteA[j] = tile_byte(sla.row_of(AKC ? 2 * j : 4 * j), sla.k_of(AKC ? 0 : 4 * j));
            byteB[j] = tile_byte(slb.row_of(BKC ? 2 * j : 4 * j), slb.k_of(BKC ? 0 : 4 * j));
        }
        Unit u{};
        int i = 0;
        bool more = unit_of(p, 0, u);
        int st = u.s0;
        float2 va[8], vb[8];
        int rb[BKC ? 4 : 1];
        auto rows = [&]() {
#pragma unroll
            for (int j = 0; j < (BKC ? 4 : 1); ++j)
                rb[j] = row_of_column(p, min(u.n0 + slb.row_of(2 * j), u.n1 - 1));
        };
        auto load = [&]() {
            int ra[AKC ? 4 : 1];
#pragma unroll
            for (int j = 0; j < (AKC ? 4 : 1); ++j) ra[j] = min(u.m0 + sla.row_of(2 * j), p.M - 1);
            load8<AKC>(va, p.A, p.A.p + u.z * p.A.sb, ra, sla, st);
            load8<BKC>(vb, p.B, p.B.p + u.z * p.B.sb, rb, slb, st);
            if (p.dk) {
                const float* w = p.dk + (int64_t)u.z * p.sdb;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = st * kStep + sla.k_of(j);
                    const float f = k < p.A.kvalid ? __ldg(&w[k]) : 0.f;
                    va[j].x *= f;
                    va[j].y *= f;
                }
            }
        };
        if (more) {
            rows();
            load();
        }
        int s = 0;
        uint32_t ph = 0;
#pragma unroll 1
        while (more) {
            if (!wait(&empty[s], ph ^ 1)) break;
            const uint32_t stage = smem_u32(smem + s * kStage);
            if (p.conjA)
#pragma unroll
                for (int j = 0; j < 8; ++j) va[j].y = -va[j].y;
            if (p.conjB)
#pragma unroll
                for (int j = 0; j < 8; ++j) vb[j].y = -vb[j].y;
            store8<AKC, false>(va, stage, byteA, sla, p.nt);
            store8<BKC, true>(vb, stage, byteB, slb, p.nt);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[s]);
            if (++s == kStages) {
                s = 0;
                ph ^= 1;
            }
            if (++st == u.s1) {
                more = unit_of(p, ++i, u);
                st = u.s0;
                if (more) rows();
            }
            if (more) load();
        }
    } else {
        // ---------------- add the finished chunks
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsAdd));
        const int c0 = (warp - kCut >> 2) * 64;               // first column of this warp's sums
        const uint32_t tq = tbase + ((uint32_t)((warp & 3) * 32) << 16) + c0;
        uint64_t acc[2][4][8];                                // [Re, Im][column group][pairs of columns]
        int a = 0;
        uint32_t aph = 0;
        bool ok = true;
        Unit u;
#pragma unroll 1
        for (int i = 0; ok && unit_of(p, i, u); ++i) {
#pragma unroll
            for (int j = 0; j < 64; ++j) acc[j >> 5][j >> 3 & 3][j & 7] = 0;
#pragma unroll 1
            for (int st = u.s0; st < u.s1; ++st) {
                if (!wait(&acc_full[a], aph)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t tr = tq + (uint32_t)(a * 256);
                if (c0 + 48 < p.nt) {
#pragma unroll
                    for (int g = 0; g < 8; ++g) add16(acc[g >> 2][g & 3], tr + (g >> 2) * p.nt + 16 * (g & 3));
                } else {
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        if (c0 + 16 * (g & 3) < p.nt) add16(acc[g >> 2][g & 3], tr + (g >> 2) * p.nt + 16 * (g & 3));
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[a]);
                if (++a == 2) {
                    a = 0;
                    aph ^= 1;
                }
            }
            const int m = u.m0 + (warp & 3) * 32 + lane;
            if (!ok || m >= p.M) continue;
            const int n0 = u.n0 + c0, n1 = u.n1 - n0;          // this warp's columns
            float2* o;
            bool vec = false;
            if (p.ksplit > 1) {
                o = p.part + (((int64_t)u.ks * p.batch + u.z) * p.M + m) * p.cols + n0;
            } else {
                o = p.C + out_at(p, u.z, m, n0);
                vec = p.vecC;
            }
#pragma unroll
            for (int g = 0; g < 4; ++g)
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int n = 16 * g + 2 * j;
                    const float2 re = unpack2(acc[0][g][j]), im = unpack2(acc[1][g][j]);
                    if ((p.ep_B > 0 || p.scn != 1) && p.ksplit == 1) {
                        if (n < n1) p.C[out_at(p, u.z, m, n0 + n)] = make_float2(re.x, im.x);
                        if (n + 1 < n1) p.C[out_at(p, u.z, m, n0 + n + 1)] = make_float2(re.y, im.y);
                    } else if (vec && n + 1 < n1) {
                        *reinterpret_cast<float4*>(o + n) = make_float4(re.x, im.x, re.y, im.y);
                    } else {
                        if (n < n1) o[n] = make_float2(re.x, im.x);
                        if (n + 1 < n1) o[n + 1] = make_float2(re.y, im.y);
                    }
                }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kIssuer) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(kTmemCols));
    }
}

// C from the parts of a split k range, added in order
__global__ void __launch_bounds__(256) cgemm_sum_kernel(const CGemmF32 p) {
    const int64_t n_el = (int64_t)p.batch * p.M * p.cols;
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n_el) return;
    const int n = (int)(i % p.cols);
    const int64_t zm = i / p.cols;
    const int m = (int)(zm % p.M), z = (int)(zm / p.M);
    if (p.tri && n < m / 128 * 128 / p.nt * p.nt) return;     // tiles left of the diagonal's are not computed
    float2 v = p.part[i];
    for (int k = 1; k < p.ksplit; ++k) {
        const float2 w = p.part[(int64_t)k * n_el + i];
        v.x += w.x;
        v.y += w.y;
    }
    p.C[out_at(p, z, m, n)] = v;
}

template <bool AKC, bool BKC>
cudaError_t launch(const CGemmF32& p, cudaStream_t s) {
    static std::atomic<bool> attr{false};
    const cudaError_t e = bip_set_once(attr, [&] {
        // the register split needs the launch to hold what it was written for
        cudaFuncAttributes at;
        cudaError_t q = cudaFuncGetAttributes(&at, cgemm_f32_kernel<AKC, BKC>);
        if (q == cudaSuccess && at.numRegs != kRegsLaunch) q = cudaErrorInvalidConfiguration;
        if (q != cudaSuccess) return q;
        return cudaFuncSetAttribute(cgemm_f32_kernel<AKC, BKC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kSmem);
    });
    if (e != cudaSuccess) return e;
    cgemm_f32_kernel<AKC, BKC><<<p.units < num_sms() ? p.units : num_sms(), kThreads, kSmem, s>>>(p);
    return cudaGetLastError();
}

bool aligned2(const void* q, int64_t a, int64_t b, int64_t c) {
    return (reinterpret_cast<uintptr_t>(q) & 15) == 0 && ((a | b | c) & 1) == 0;
}

}  // namespace

// Tile widths, the k split and the workspace (float2 elements of `part`).
// A chunk of a tile takes about 2800 clocks whatever the tile's width (48, 104
// and 128 columns measured: the cutting warps' chain), so the columns go into
// as few tiles as they fill; the coupling's columns are taken through all
// channels without the padding between them (3 channels of 193 beams: 5 tiles
// where channel by channel takes 6).  Callers put the side with few rows on the
// columns, since rows are padded to 128.  The split: the parts
// that minimise rounds x (chunks per part + the pipeline's fill, about three
// chunks), plus the parts' way through memory at about 2.5 KB per clock.  It
// is chosen for plan_batch entries and plan_rows rows, so that a site's sums do
// not depend on how full its batch is, nor a beam's on its cube's chunks.
cudaError_t bip_cgemm_plan(CGemmF32& p, size_t* part_elems) {
    if (p.M < 1 || p.N < 1 || p.batch < 1) return cudaErrorInvalidValue;
    for (CGemmOperand* o : {&p.A, &p.B}) {
        if (o->kvalid < 1 || o->nper < 1) return cudaErrorInvalidValue;
        o->kper = (o->kvalid + kStep - 1) / kStep * kStep;
        o->vec = o->sk == 1 && aligned2(o->p, o->sr, o->sk2, o->sb);
        if (o->sk != 1 && o->sr != 1) return cudaErrorInvalidValue;
        // a row's length and offsets within a chunk are 32-bit in the kernel
        if (o->sr > 0x7fffffff || kStep * o->sk > 0x7fffffff) return cudaErrorInvalidValue;
    }
    if (p.A.kvalid != p.B.kvalid || p.A.nper != p.B.nper) return cudaErrorInvalidValue;
    if (p.dk && p.A.nper != 1) return cudaErrorInvalidValue;
    p.vecC = p.scn == 1 && aligned2(p.C, p.scm, p.scb, 0) ? 1 : 0;
    if (p.ep_B > 0 && (p.ep_n < 1 || p.ep_n > p.ep_B || p.N % p.ep_B)) return cudaErrorInvalidValue;
    p.cols = p.ep_B > 0 ? p.N / p.ep_B * p.ep_n : p.N;
    p.n_tiles = (p.cols + 127) / 128;
    p.nt = ((p.cols + p.n_tiles - 1) / p.n_tiles + 7) / 8 * 8;
    p.n_tiles = (p.cols + p.nt - 1) / p.nt;
    const int m_tiles = (p.M + 127) / 128;
    p.tiles = 0;
    for (int mt = 0; mt < m_tiles; ++mt) p.tiles += std::max(0, p.n_tiles - (p.tri ? mt * 128 / p.nt : 0));
    p.steps = p.A.nper * (p.A.kper / kStep);
    const int pb = p.plan_batch > 0 ? p.plan_batch : p.batch;
    if ((int64_t)p.tiles * std::max(pb, p.batch) * 16 > (1 << 26)) return cudaErrorInvalidValue;
    const int rows = p.plan_rows > 0 ? p.plan_rows : p.M;
    const int64_t units = (p.plan_rows > 0 ? (int64_t)((rows + 127) / 128) * p.n_tiles : p.tiles) * pb;
    const int sms = num_sms();
    const double chunk = 2800.0;                               // clocks, whatever the width
    const double bytes = 8.0 * pb * (double)rows * p.cols;
    double best = 0.0;
    p.ksplit = 1;
    for (int S = 1; S <= 16 && S * 4 <= p.steps; ++S) {
        const double rounds = (double)((units * S + sms - 1) / sms);
        double t = rounds * ((p.steps + S - 1) / S + 3) * chunk;
        if (S > 1) t += (2.0 * S + 1.0) * bytes / 2500.0 + 6000.0;
        if (S == 1 || t < best) {
            best = t;
            p.ksplit = S;
        }
    }
    p.units = p.tiles * p.batch * p.ksplit;
    *part_elems = p.ksplit > 1 ? (size_t)p.ksplit * p.batch * p.M * p.cols : 0;
    return cudaSuccess;
}

cudaError_t bip_cgemm_f32(const CGemmF32& p, cudaStream_t s) {
    if (p.units < 1 || p.nt < 8 || p.nt > 128 || p.nt % 8 || !p.err || (p.ksplit > 1 && !p.part))
        return cudaErrorInvalidValue;
    const bool a = p.A.sk == 1, b = p.B.sk == 1;
    cudaError_t e = a && b ? launch<true, true>(p, s)
                  : a      ? launch<true, false>(p, s)
                  : b      ? launch<false, true>(p, s)
                           : launch<false, false>(p, s);
    if (e != cudaSuccess || p.ksplit == 1) return e;
    const int64_t n = (int64_t)p.batch * p.M * p.cols;
    cgemm_sum_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p);
    return cudaGetLastError();
}
