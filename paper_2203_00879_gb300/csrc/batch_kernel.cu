// One persistent launch per RK step for all boxes of a context (mixed form).
//
// A box's RK4 step is a chain of phases -- per stage the x, y and z flux
// sweeps (Sec. 3), the fused viscous / source / RK kernel (Sec. 2, Sec. 4) and
// the wall conditions -- and each phase is a
// set of independent blocks: the blocks the stand-alone kernels would launch.
// Here one kernel runs them all.  The host lists work items (box, stage,
// phase, a run of blocks), each box's phases in order; every block of the
// persistent grid takes the next item from an atomic counter, waits until the
// box's previous phase has completed all its items, runs the item's blocks
// with the same device code as the stand-alone kernels (sweep32.cuh,
// visc_body.cuh, wall_body.cuh), and counts the item done.  Boxes advance
// independently, so small boxes fill the GPU side by side without a launch
// per kernel and box.
//
// An item only ever waits for items listed before it, which blocks that were
// already running took, so the grid needs no co-residency to make progress.
// Each wait is bounded (globaltimer): when it gives up it sets the batch's
// abort word and the context's error word (the host reports NOPCS_ETIMEOUT),
// every later wait returns at once, and the kernel ends.  The completion
// counters use release / acquire at GPU scope; the data of a finished phase is
// read by plain (coherent) loads after the acquiring thread's barrier.
#include <algorithm>
#include <string>
#include <vector>

#include "sweep32.cuh"
#include "visc_body.cuh"
#include "wall_body.cuh"

namespace nopcs {

namespace {

constexpr int BT = 256;             // threads per block (the viscous tile's)
// Lines per tile of the y and z sweeps (half as many with a ring of 8 groups)
// and rows of theirs in flight, at two blocks per SM: a step of the 64-box
// workload takes 39.4 ms, of one 256^3 box 9.1 ms; with 160 lines 39.4 and 9.8,
// with 160 lines and 8 rows 42.2 and 10.7, at three blocks per SM (80 registers
// a thread, the sweeps spill) with 96 lines and 2 rows 46.5 and 11.6.  (All
// before the stage and wall kernels were changed: now 36.2 and 8.5.)
constexpr int BMARCH = 128, BU = 4;
// wall nodes per tile: four passes of a block, so that a box's wall phase
// spreads over many blocks instead of holding the box's next phase behind a few
// long items
constexpr unsigned WALL_CHUNK = 4 * BT;
enum { PH_SX = 0, PH_SY, PH_SZ, PH_VISC, PH_WALL, NPH };

struct BStage {
    Sweep32Args sw[3];
    VArgs<float> va;
    double *Q;  // wall conditions: the FP64 state (stage 4) or null (stage state Ww)
    float *Dn, *Wf, *Ww;
};

struct BBox {
    BoxDev bx;
    int ntile[NPH];  // blocks of the stand-alone launch per phase
    int chunk[NPH];  // blocks per item
    int nitem[NPH];  // items per phase
    int gx, gy;      // viscous grid in x and y
    BStage st[4];
};

struct BItem {
    int box, stage, phase, first;
};

struct BParams {
    const BBox *boxes;
    const BItem *items;
    int nitems;
    int *next;   // work counter
    int *abort;  // set when a wait gave up
    int *done;   // [box][stage][phase] finished items
    int *err;    // the context's error word (2: a wait gave up)
    unsigned long long wait_ns;
    int withhold;  // test: box 0's first dependency needs one item more than exists
};

__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_add(int *p, int v)
{
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait until *ctr >= need, at most wait_ns; false if the wait gave up or the
// batch was aborted.
__device__ bool wait_at_least(const BParams &p, const int *ctr, int need)
{
    const unsigned long long t0 = now_ns();
    for (;;) {
        if (ld_acquire(ctr) >= need) return true;
        if (ld_acquire(p.abort) != 0) return false;
        if (now_ns() - t0 > p.wait_ns) {
            atomicExch(p.abort, 1);
            atomicCAS(p.err, 0, 2);
            return false;
        }
        __nanosleep(256);
    }
}

// The phase bodies are separate (not inlined) functions, so that each gets the
// kernel's whole register budget instead of all of them sharing one
// allocation inside the item loop.
__device__ __noinline__ void run_sweep_x(const Sweep32Args &a, int v, float *sm)
{
    const int w = (int)(threadIdx.x >> 5);
    scan_any<MODE_FLUX>(a, v * (BT / 32) + w, sm + w * SweepMode<MODE_FLUX>::NF * SC_FS);
}
template <int AXIS>
__device__ __noinline__ void run_march(const Sweep32Args &a, int v, float *sm)
{
    if (threadIdx.x >= BMARCH) return;
    if (a.ring == 8) {
        if (threadIdx.x >= BMARCH / 2) return;
        if (a.ga == AXIS)
            march_body<MODE_FLUX, AXIS, true, 8, BMARCH / 2, BU, false>(a, (unsigned)v, (int)threadIdx.x, sm);
        else
            march_body<MODE_FLUX, AXIS, false, 8, BMARCH / 2, BU, false>(a, (unsigned)v, (int)threadIdx.x, sm);
    } else {
        if (a.ga == AXIS)
            march_body<MODE_FLUX, AXIS, true, 4, BMARCH, BU, false>(a, (unsigned)v, (int)threadIdx.x, sm);
        else
            march_body<MODE_FLUX, AXIS, false, 4, BMARCH, BU, false>(a, (unsigned)v, (int)threadIdx.x, sm);
    }
}
// the viscous stage kernel in the specialisations of the stand-alone launch
template <class S>
__device__ __noinline__ void run_visc(const VArgs<float> &va, int bx, int by, int bz, unsigned char *sm)
{
    visc_rk_block<float, S>(va, bx, by, bz, sm);
}
template <int GA>
__device__ __forceinline__ void run_visc_ga(const VArgs<float> &va, int bx, int by, int bz, unsigned char *sm)
{
    switch (va.stage) {
    case 1: run_visc<Spec<1, GA>>(va, bx, by, bz, sm); return;
    case 2: run_visc<Spec<2, GA>>(va, bx, by, bz, sm); return;
    case 3: run_visc<Spec<3, GA>>(va, bx, by, bz, sm); return;
    default: run_visc<Spec<4, GA>>(va, bx, by, bz, sm);
    }
}
__device__ __forceinline__ void run_visc_any(const VArgs<float> &va, int bx, int by, int bz, unsigned char *sm)
{
    if (va.ga == 2)
        run_visc_ga<2>(va, bx, by, bz, sm);
    else
        run_visc_ga<-1>(va, bx, by, bz, sm);
}

__global__ void __launch_bounds__(BT, 2) batch_step_kernel(const BParams p)
{
    extern __shared__ __align__(32) unsigned char smraw[];
    __shared__ int s_item, s_go;
    // the item's arguments, copied from the device box table: the phase code
    // then reads its pointers and constants from shared memory instead of
    // through global loads ahead of every data access
    constexpr int ARGW =
        (int)((sizeof(VArgs<float>) > sizeof(Sweep32Args) ? sizeof(VArgs<float>) : sizeof(Sweep32Args)) / 8);
    static_assert(sizeof(VArgs<float>) % 8 == 0 && sizeof(Sweep32Args) % 8 == 0, "copied in 8-byte words");
    __shared__ unsigned long long s_args[ARGW];
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(p.next, 1);
        __syncthreads();
        const int i = s_item;
        if (i >= p.nitems) return;
        const BItem it = p.items[i];
        const BBox &B = p.boxes[it.box];
        if (threadIdx.x == 0) {
            // the previous phase of this box (of the previous stage for the
            // first phase of a stage)
            int ds = it.stage, dp = it.phase - 1;
            if (dp < 0) {
                ds -= 1;
                dp = NPH - 1;
            }
            bool ok = ld_acquire(p.abort) == 0;
            if (ok && ds >= 0) {
                const int need = B.nitem[dp] + (p.withhold && it.box == 0 && ds == 0 && dp == PH_SX ? 1 : 0);
                ok = wait_at_least(p, p.done + (it.box * 4 + ds) * NPH + dp, need);
            }
            s_go = ok;
            // acquire at GPU scope before the block's barrier: the block's
            // plain loads after it see the finished phase's data (the L1 lines
            // of this SM are not left stale by it); the whole block's loads
            // going to L2 only instead (-dlcm=cg) gave the same bits and was
            // three times slower
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
        }
        __syncthreads();
        if (s_go) {
            const BStage &S = B.st[it.stage];
            Sweep32Args *ssw = reinterpret_cast<Sweep32Args *>(s_args);
            VArgs<float> *sva = reinterpret_cast<VArgs<float> *>(s_args);
            {
                auto copy = [&](void *dst, const void *src, int bytes) {
                    const unsigned long long *a = (const unsigned long long *)src;
                    unsigned long long *b = (unsigned long long *)dst;
                    for (int k = threadIdx.x; k < bytes / 8; k += BT) b[k] = a[k];
                };
                if (it.phase <= PH_SZ) {
                    copy(ssw, &S.sw[it.phase], (int)sizeof(Sweep32Args));
                } else if (it.phase == PH_VISC) {
                    copy(sva, &S.va, (int)sizeof(VArgs<float>));
                }
                __syncthreads();
            }
            const int last = min(it.first + B.chunk[it.phase], B.ntile[it.phase]);
            for (int v = it.first; v < last; ++v) {
                switch (it.phase) {
                case PH_SX: run_sweep_x(*ssw, v, reinterpret_cast<float *>(smraw)); break;
                case PH_SY: run_march<1>(*ssw, v, reinterpret_cast<float *>(smraw)); break;
                case PH_SZ: run_march<2>(*ssw, v, reinterpret_cast<float *>(smraw)); break;
                case PH_VISC: run_visc_any(*sva, v % B.gx, (v / B.gx) % B.gy, v / (B.gx * B.gy), smraw); break;
                default: {  // the walls, block 0 the corners
                    if (v == 0) {
                        corner_block(B.bx, threadIdx.x, S.Q, S.Dn, S.Wf, S.Ww);
                        break;
                    }
                    const unsigned t1 = min(wall_count(B.bx), (unsigned)v * WALL_CHUNK);
                    for (unsigned t = (unsigned)(v - 1) * WALL_CHUNK + threadIdx.x; t < t1; t += BT)
                        wall_node(B.bx, t, S.Q, S.Dn, S.Wf, S.Ww);
                }
                }
                __syncthreads();  // the next block of the item reuses the shared memory
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            red_release_add(p.done + (it.box * 4 + it.stage) * NPH + it.phase, 1);
        }
    }
}

}  // namespace

struct BatchPlan {
    void *mem = nullptr;      // boxes, items, counters
    BParams p{};
    int grid = 0;
    size_t smem = 0;
    size_t counter_bytes = 0;
    int *counters = nullptr;  // next, abort, done[]
};

cudaError_t batch_plan_build(const std::vector<BatchBoxIn> &in, BatchPlan **out, std::string &msg)
{
    *out = nullptr;
    const int nb = (int)in.size();
    std::vector<BBox> boxes(nb);
    std::vector<BItem> items;
    constexpr int NF = SweepMode<MODE_FLUX>::NF;
    const size_t smem = std::max({visc_smem<float>(), scan_smem(NF, BT / 32), march_smem(NF, 4, BMARCH)});
    for (int b = 0; b < nb; ++b) {
        const BatchBoxIn &I = in[b];
        BBox &B = boxes[b];
        B.bx = I.bx;
        for (int s = 1; s <= 4; ++s) {
            BStage &S = B.st[s - 1];
            const float *Win = I.W[(s - 1) & 1];
            float *Wout = I.W[s & 1];
            for (int a = 0; a < 3; ++a) {
                // the stand-alone launch's pieces (the same arithmetic)
                Sweep32Args &w = S.sw[a];
                w = Sweep32Args{};
                if (!flux32_args(I.op[a], a, I.bx, Win, I.R, w)) {
                    msg = "a flux sweep of a box does not fit the batched kernel's blocks";
                    return cudaErrorInvalidConfiguration;
                }
                const long long per = SC_USE * (BT / 32), bm = w.ring == 8 ? BMARCH / 2 : BMARCH;
                B.ntile[PH_SX + a] = (int)(a == 0 ? (w.tot + per - 1) / per
                                                  : (w.cols + bm - 1) / bm * w.nseg);
            }
            StageRegs<float> r;
            r.Qn = I.Qn;
            r.Kacc = I.K;
            r.Dn = I.Dn;
            r.Wn = Wout;
            S.va = make_vargs<float>(I.bx, Win, I.R, s, r);
            const dim3 vg = visc_grid<float>(I.bx, S.va.zc);
            B.gx = (int)vg.x;
            B.gy = (int)vg.y;
            B.ntile[PH_VISC] = (int)(vg.x * vg.y * vg.z);
            if (s < 4) {
                S.Q = nullptr;
                S.Dn = nullptr;
                S.Wf = nullptr;
                S.Ww = Wout;
            } else {
                S.Q = I.Qn;
                S.Dn = I.Dn;
                S.Wf = Wout;
                S.Ww = nullptr;
            }
        }
        B.ntile[PH_WALL] = 1 + (int)((wall_count(I.bx) + WALL_CHUNK - 1) / WALL_CHUNK);
        // blocks per item: about a quarter of a GPU wave per phase of a big
        // box, single blocks for small ones
        for (int ph = 0; ph < NPH; ++ph) {
            const int nt = B.ntile[ph] > 0 ? B.ntile[ph] : 1;
            int ch = nt / (152 * 3 * 16);
            B.chunk[ph] = ch < 1 ? 1 : ch;
            B.nitem[ph] = (nt + B.chunk[ph] - 1) / B.chunk[ph];
        }
    }
    // Items on diagonals: box b's phase g (= stage x NPH + phase) on diagonal
    // g + b, diagonals in order, boxes in order within one.  Every box's
    // phases stay in order (the dependency rule), and consecutive phases of a
    // box are a whole diagonal apart: while a block waits for box b's
    // previous phase, the items behind it belong to other boxes at other
    // phases, whose dependencies are older.  (Stage-major order, every box at
    // the same phase, left blocks waiting at each phase boundary.)
    for (int d = 0; d < 4 * NPH + nb - 1; ++d)
        for (int b = 0; b < nb; ++b) {
            const int g = d - b;
            if (g < 0 || g >= 4 * NPH) continue;
            const int s = g / NPH, ph = g % NPH;
            for (int k = 0; k < boxes[b].nitem[ph]; ++k) items.push_back(BItem{b, s, ph, k * boxes[b].chunk[ph]});
        }
    if (smem > 227 * 1024) {
        msg = "the batched kernel's blocks need more shared memory than a block can have";
        return cudaErrorInvalidConfiguration;
    }
    BatchPlan *P = new BatchPlan();
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t bb = al(sizeof(BBox) * nb), ib = al(sizeof(BItem) * items.size());
    P->counter_bytes = sizeof(int) * (2 + (size_t)nb * 4 * NPH);
    cudaError_t e = dev_alloc(&P->mem, bb + ib + P->counter_bytes);
    if (e != cudaSuccess) {
        delete P;
        return e;
    }
    char *base = (char *)P->mem;
    e = cudaMemcpy(base, boxes.data(), sizeof(BBox) * nb, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(base + bb, items.data(), sizeof(BItem) * items.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int per_sm = 0, nsm = 0, dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_step_kernel, BT, smem);
    if (e != cudaSuccess || per_sm < 1) {
        dev_free(P->mem);
        delete P;
        msg = "the batched kernel does not fit an SM";
        return e != cudaSuccess ? e : cudaErrorInvalidConfiguration;
    }
    P->counters = (int *)(base + bb + ib);
    P->p.boxes = (const BBox *)base;
    P->p.items = (const BItem *)(base + bb);
    P->p.nitems = (int)items.size();
    P->p.next = P->counters;
    P->p.abort = P->counters + 1;
    P->p.done = P->counters + 2;
    P->grid = per_sm * nsm < P->p.nitems ? per_sm * nsm : P->p.nitems;
    P->smem = smem;
    *out = P;
    return cudaSuccess;
}

cudaError_t batch_launch(BatchPlan *P, int *err, double wait_s, int withhold, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(P->counters, 0, P->counter_bytes, st);
    if (e != cudaSuccess) return e;
    BParams p = P->p;
    p.err = err;
    p.wait_ns = (unsigned long long)(wait_s * 1e9);
    p.withhold = withhold;
    batch_step_kernel<<<P->grid, BT, P->smem, st>>>(p);
    return cudaGetLastError();
}

void batch_plan_free(BatchPlan *P)
{
    if (!P) return;
    if (P->mem) dev_free(P->mem);
    delete P;
}

int batch_plan_items(const BatchPlan *P) { return P ? P->p.nitems : 0; }

}  // namespace nopcs
