// Batched intensity sweep: several independent slabs (uneven sizes, particle counts and laser
// intensities) advanced together. Each slab is an ordinary context (pic_init on a slice of the
// batch workspace); a step of the whole batch is
//   k_particles_batch    one persistent launch over the tiles of every slab
//   k_fields_batch       the field update of every slab, which also prepares the next step (clears
//                        its currents, starts its node density, evaluates its antenna scalars)
// (the transport stage, and slabs with one set of grids, have k_prepare_batch in front instead) and is
// recorded once as a CUDA graph per parity of the double-buffered grids, then replayed. The per-slab
// arguments live in device memory (copied into a constant-memory table in front of the particle kernel), so
// a cell sort (host-driven, every sort_every steps) only refreshes them; the graphs stay valid.
#include <cstring>
#include <new>
#include <vector>

#include "pic_internal.cuh"

namespace gbpic {
void sort_species_impl(Ctx& c, int s, cudaStream_t st, int from_b, int64_t* launches);
int max_batch_slabs();

constexpr int kMaxSlabs = 48;    // the constant-memory argument table of the batched particle kernel
static_assert(kMaxSlabs <= kMaxFieldSlabs, "every slab's field arguments fit the batched field kernels' parameters");

// Clears the currents a step deposits into (the transport stage has none) and starts the next node
// density from the current one.
__global__ void k_prepare_batch(const StepArgs* __restrict__ args)
{
    const StepArgs& a = args[blockIdx.y];
    const size_t nn = (size_t)(a.nz + 1) * a.nx;
    for (size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x; j < nn; j += (size_t)gridDim.x * blockDim.x) {
        if (a.full) {
            a.J[0][j] = 0;
            a.J[1][j] = 0;
            a.J[2][j] = 0;
        }
        a.rho_next[j] = a.rho_cur[j];
    }
}

}  // namespace gbpic

using namespace gbpic;

struct pic_batch {
    int n;
    pic_ctx* slab[kMaxSlabs];
    cudaStream_t st;
    int full, twin, pot, minW, maxW, nsm, sort_every;     // twin: two sets of grids (full mode)
    size_t max_nn;
    StepArgs* args_dev;          // [2][n]: parity 0 (density in buffer 0) and parity 1
    FieldBatch fields[2];        // every slab's field arguments per parity (host copy, passed by value)
    AntennaParams* ap_dev;       // [n]
    long long* step_dev;         // [n]
    float* ant_dev;              // [2][n][2]: the antenna scalars of a step of each parity
    WorkItem* items;             // work items of every slab's tiles, rebuilt after a sort
    int* nitems;
    int items_cap;
    cudaGraphExec_t graph[2];
    int captured;
    int timing;
    cudaEvent_t ev[6];
    double ms[3];
    int64_t nlaunch[4];
    int sticky;
};

namespace {

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

int64_t batch_items_cap(const pic_config* cfgs, int n)
{
    int64_t t = 0;
    for (int s = 0; s < n; s++) t += work_item_cap_of(&cfgs[s]);
    return t;
}

size_t batch_tail_bytes(const pic_config* cfgs, int n)
{
    return a256(sizeof(WorkItem) * (size_t)batch_items_cap(cfgs, n)) + a256(4) +
           a256(sizeof(StepArgs) * 2 * n) + a256(sizeof(AntennaParams) * n) + a256(8 * (size_t)n) +
           a256(16 * (size_t)n);
}

// The other parity of a slab's double-buffered grids (density; with fields also the fields and the
// currents, which a step swaps too).
void flip_parity(Ctx& c)
{
    c.cur = 1 - c.cur;
    if (!c.Jn[0]) return;
    swap_currents(c);
    swap_fields(c);
}

// Arguments of a step that starts at parity p: the particle kernel deposits into the cleared
// currents Jn and the field update then reads them (as J).
int upload_args(pic_batch* b)
{
    std::vector<StepArgs> h(2 * b->n);
    for (int s = 0; s < b->n; s++) {
        Ctx& c = b->slab[s]->c;
        for (int k = 0; k < 2; k++) {
            const int p = c.cur;
            StepArgs& a = h[p * b->n + s];
            a = make_step_args(c);
            for (int q = 0; q < 3 && c.Jn[0]; q++) a.J[q] = c.Jn[q];
            flip_parity(c);
        }
    }
    if (cudaMemcpyAsync(b->args_dev, h.data(), sizeof(StepArgs) * h.size(), cudaMemcpyHostToDevice, b->st) !=
        cudaSuccess)
        return PIC_ECUDA;
    return cudaStreamSynchronize(b->st) == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

void enqueue_prepare(pic_batch* b, int parity)
{
    dim3 pg((unsigned)((b->max_nn + 1023) / 1024 > 4096 ? 4096 : (b->max_nn + 1023) / 1024), b->n);
    k_prepare_batch<<<pg, 256, 0, b->st>>>(b->args_dev + parity * b->n);
}

void enqueue_step(pic_batch* b, int parity)
{
    const StepArgs* args = b->args_dev + parity * b->n;
    if (!b->twin) enqueue_prepare(b, parity);
    if (b->full && !b->twin)
        launch_antenna_batch(b->ap_dev, b->step_dev, b->ant_dev + parity * 2 * b->n, b->n, b->st);
    if (b->timing) cudaEventRecord(b->ev[0], b->st);
    launch_particle_step_batch(args, b->n, b->items, b->nitems, b->full, b->pot, b->minW, b->maxW, b->nsm, b->st);
    if (b->timing) cudaEventRecord(b->ev[1], b->st);
    if (b->twin) {
        launch_fields_batch(b->fields[parity], b->ap_dev, b->step_dev, b->ant_dev + (1 - parity) * 2 * b->n, b->st);
    } else if (b->full) {
        for (int s = 0; s < b->n; s++) launch_fields_one_set(b->fields[parity].f[s], b->st);
        launch_step_done(b->step_dev, b->n, b->st);
    }
    if (b->timing) cudaEventRecord(b->ev[2], b->st);
}

// Kernels of a step: particles and fields, or prepare and particles (transport), or with one set of grids those, the
// antenna's, three per slab and the counters'.
int launches(const pic_batch* b) { return b->full && !b->twin ? 4 + 3 * b->n : 2; }

// One list of work items over every slab's tiles, after a sort or a slab's state was written.
void build_items(pic_batch* b)
{
    int64_t n = 0;
    for (int s = 0; s < b->n; s++) {
        const Ctx& c = b->slab[s]->c;
        n += c.sp[0].n + (c.nsp > 1 ? c.sp[1].n : 0);
    }
    cudaMemsetAsync(b->nitems, 0, sizeof(int), b->st);
    const int chunk = item_chunk(n, particle_slots(b->nsm, b->full, 1, b->maxW));
    for (int s = 0; s < b->n; s++) {
        launch_work_items(b->slab[s]->c, s, chunk, b->items, b->nitems, b->items_cap, b->st);
        b->slab[s]->c.items_ok = 1;
    }
}

// The fields' update prepares the step after it; the first step, and one after a slab's state was
// written from outside (a checkpoint, new particles), is prepared here. A slab sorted on its own has
// changed its two particle buffers over, and a restored one is at its checkpoint's step: the arguments
// and the counters of the laser pulse are taken from the slabs.
int prepare(pic_batch* b)
{
    bool ready = true, listed = true;
    long long step[kMaxSlabs];
    for (int s = 0; s < b->n; s++) {
        const Ctx& c = b->slab[s]->c;
        listed &= c.items_ok != 0;
        ready &= c.prepared != 0;
        step[s] = (long long)c.step;
    }
    if (!listed) {
        const int r = upload_args(b);
        if (r) return r;
        build_items(b);
    }
    if (!b->full || ready) return PIC_OK;
    // a pageable source: the call returns once the counters have been staged
    if (cudaMemcpyAsync(b->step_dev, step, 8 * (size_t)b->n, cudaMemcpyHostToDevice, b->st) != cudaSuccess)
        return PIC_ECUDA;
    if (!b->twin) return PIC_OK;             // every step prepares itself
    const int parity = b->slab[0]->c.cur;
    enqueue_prepare(b, parity);
    launch_antenna_batch(b->ap_dev, b->step_dev, b->ant_dev + parity * 2 * b->n, b->n, b->st);
    b->nlaunch[3] += 2;
    return PIC_OK;
}

// Steps since the last sort of the slab sorted longest ago (a restored slab brings its own count).
int steps_since_sort(const pic_batch* b)
{
    int n = 0;
    for (int s = 0; s < b->n; s++) n = b->slab[s]->c.steps_since_sort > n ? b->slab[s]->c.steps_since_sort : n;
    return n;
}

int capture(pic_batch* b)
{
    for (int p = 0; p < 2; p++) {
        cudaGraph_t g;
        if (cudaStreamBeginCapture(b->st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return PIC_ECUDA;
        enqueue_step(b, p);
        if (cudaStreamEndCapture(b->st, &g) != cudaSuccess) return PIC_ECUDA;
        const cudaError_t e = cudaGraphInstantiate(&b->graph[p], g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return PIC_ECUDA;
    }
    b->captured = 1;
    return PIC_OK;
}

}  // namespace

// Bytes of the batch; *twin: the slabs have two sets of grids, which all of them have or none (kTwinBytes for all).
static int batch_bytes(const pic_config* cfgs, int n, bool* twin, size_t* bytes)
{
    size_t t = 0;
    bool all = true;
    for (int s = 0; s < n; s++) {
        size_t b = 0;
        bool two = *twin;
        const int r = workspace_bytes(&cfgs[s], &two, &b);
        if (r) return r;
        all &= two;
        t += a256(b);
    }
    if (*twin && cfgs[0].mode == PIC_MODE_FULL && (!all || t > kTwinBytes)) {
        *twin = false;
        return batch_bytes(cfgs, n, twin, bytes);
    }
    *twin = all;
    *bytes = t + batch_tail_bytes(cfgs, n);
    return PIC_OK;
}

extern "C" {

int pic_batch_workspace_size(const pic_config* cfgs, int32_t n, size_t* bytes)
{
    if (!cfgs || !bytes || n < 1 || n > kMaxSlabs) return PIC_EINVAL;
    for (int s = 0; s < n; s++) {
        if (cfgs[s].mode != cfgs[0].mode || (cfgs[s].dims != 0 && cfgs[s].dims != 2)) return PIC_EINVAL;
        if (cfgs[s].pot_mode != cfgs[0].pot_mode || cfgs[s].lattice != cfgs[0].lattice)
            return PIC_EINVAL;   // one kernel instance
    }
    if (batch_items_cap(cfgs, n) >= (1LL << 31)) return PIC_EINVAL;
    bool twin = true;
    return batch_bytes(cfgs, n, &twin, bytes);
}

int pic_batch_init(const pic_config* cfgs, int32_t n, void* workspace, size_t bytes, void* stream, pic_batch** out)
{
    if (!out) return PIC_EINVAL;
    *out = nullptr;
    size_t need = 0;
    int r = pic_batch_workspace_size(cfgs, n, &need);
    if (r) return r;
    if (!workspace || ((uintptr_t)workspace & 255) || !stream) return PIC_EINVAL;
    if (bytes < need) return PIC_ENOMEM;
    pic_batch* b = new (std::nothrow) pic_batch();
    if (!b) return PIC_ENOMEM;
    b->n = n;
    b->st = (cudaStream_t)stream;
    char* p = (char*)workspace;
    bool twin = true;
    batch_bytes(cfgs, n, &twin, &need);
    b->twin = twin;
    for (int s = 0; s < n; s++) {
        size_t sb = 0;
        bool two = twin;
        workspace_bytes(&cfgs[s], &two, &sb);
        r = init_context(&cfgs[s], p, sb, stream, &b->slab[s], twin);
        if (r) {
            for (int q = 0; q < s; q++) pic_free(b->slab[q]);
            delete b;
            return r;
        }
        b->slab[s]->c.in_batch = 1;
        p += a256(sb);
        const Ctx& c = b->slab[s]->c;
        b->maxW = c.W > b->maxW ? c.W : b->maxW;
        b->minW = s == 0 || c.W < b->minW ? c.W : b->minW;
        b->max_nn = c.nn > b->max_nn ? c.nn : b->max_nn;
        b->nsm = c.nsm;
    }
    b->full = cfgs[0].mode == PIC_MODE_FULL;
    b->pot = pot_code(cfgs[0]);   // kernel instance
    b->sort_every = cfgs[0].sort_every;
    b->args_dev = reinterpret_cast<StepArgs*>(p);
    p += a256(sizeof(StepArgs) * 2 * n);
    b->ap_dev = reinterpret_cast<AntennaParams*>(p);
    p += a256(sizeof(AntennaParams) * n);
    b->step_dev = reinterpret_cast<long long*>(p);
    p += a256(8 * (size_t)n);
    b->ant_dev = reinterpret_cast<float*>(p);
    p += a256(16 * (size_t)n);
    b->items = reinterpret_cast<WorkItem*>(p);
    b->items_cap = (int)batch_items_cap(cfgs, n);
    p += a256(sizeof(WorkItem) * (size_t)b->items_cap);
    b->nitems = reinterpret_cast<int*>(p);
    std::vector<AntennaParams> ap(n);
    for (int s = 0; s < n; s++) {
        Ctx& c = b->slab[s]->c;
        ap[s] = make_antenna_params(c);
        if (!b->full) continue;
        for (int k = 0; k < 2; k++) {
            // the update of a step of this parity follows its moves: the density and the currents
            // are the other buffers, the fields not yet
            const int par = c.cur;
            c.cur = 1 - c.cur;
            if (twin) swap_currents(c);
            FieldArgs& f = b->fields[par].f[s];
            f = make_field_args(c);
            f.ant = b->ant_dev + par * 2 * n + 2 * s;
            c.cur = par;
            if (twin) swap_currents(c);
            flip_parity(c);
        }
    }
    for (int par = 0; par < 2; par++) {
        b->fields[par].n = n;
        if (b->twin) field_row_blocks(b->fields[par]);
    }
    const bool ok = cudaMemcpyAsync(b->ap_dev, ap.data(), sizeof(AntennaParams) * n, cudaMemcpyHostToDevice, b->st) ==
                    cudaSuccess;
    r = ok && cudaStreamSynchronize(b->st) == cudaSuccess ? PIC_OK : PIC_ECUDA;
    for (int q = 0; q < 6 && r == PIC_OK; q++)
        if (cudaEventCreate(&b->ev[q]) != cudaSuccess) r = PIC_ECUDA;
    if (r) {
        for (int q = 0; q < n; q++) pic_free(b->slab[q]);
        delete b;
        return r;
    }
    *out = b;
    return PIC_OK;
}

void pic_batch_free(pic_batch* b)
{
    if (!b) return;
    for (int p = 0; p < 2; p++)
        if (b->captured) cudaGraphExecDestroy(b->graph[p]);
    for (int q = 0; q < 6; q++)
        if (b->ev[q]) cudaEventDestroy(b->ev[q]);
    for (int s = 0; s < b->n; s++) pic_free(b->slab[s]);
    delete b;
}

int pic_batch_slab(pic_batch* b, int32_t i, pic_ctx** out)
{
    if (!b || !out || i < 0 || i >= b->n) return PIC_EINVAL;
    *out = b->slab[i];
    return PIC_OK;
}

int pic_batch_step(pic_batch* b, int32_t nsteps)
{
    if (!b || nsteps < 0) return PIC_EINVAL;
    if (b->sticky) return b->sticky;
    if (nsteps > 0) {
        const int r = prepare(b);
        if (r) return r;
    }
    for (int it = 0; it < nsteps; it++) {
        if (b->sort_every > 0 && steps_since_sort(b) >= b->sort_every) {
            if (b->timing) cudaEventRecord(b->ev[3], b->st);
            for (int s = 0; s < b->n; s++) {
                Ctx& c = b->slab[s]->c;
                for (int sp = 0; sp < c.nsp; sp++) sort_species_impl(c, sp, b->st, 0, &b->nlaunch[2]);
                c.steps_since_sort = 0;
            }
            if (b->timing) {
                cudaEventRecord(b->ev[4], b->st);
                cudaEventSynchronize(b->ev[4]);
                float ms = 0.f;
                cudaEventElapsedTime(&ms, b->ev[3], b->ev[4]);
                b->ms[2] += ms;
            }
            const int r = upload_args(b);      // the sort swapped the particle buffers
            if (r) return r;
            build_items(b);
        }
        const int parity = b->slab[0]->c.cur;
        if (b->timing) {
            // direct launches with events around the particle kernel and the field kernels
            enqueue_step(b, parity);
            if (cudaEventSynchronize(b->ev[2]) != cudaSuccess) return PIC_ECUDA;
            float m0 = 0.f, m1 = 0.f;
            cudaEventElapsedTime(&m0, b->ev[0], b->ev[1]);
            cudaEventElapsedTime(&m1, b->ev[1], b->ev[2]);
            b->ms[0] += m0;
            b->ms[1] += m1;
            b->nlaunch[0] += 1;
            b->nlaunch[1] += b->twin ? 1 : (b->full ? 3 * b->n : 0);
            b->nlaunch[3] += launches(b);
        } else {
            if (!b->captured) {
                const int r = capture(b);
                if (r) return r;
            }
            if (cudaGraphLaunch(b->graph[parity], b->st) != cudaSuccess) return PIC_ECUDA;
            b->nlaunch[3] += launches(b);
        }
        for (int s = 0; s < b->n; s++) {
            Ctx& c = b->slab[s]->c;
            flip_parity(c);
            c.prepared = c.Jn[0] != nullptr;
            c.step++;
            c.steps_since_sort++;
        }
    }
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(b->st) != cudaSuccess) return PIC_ECUDA;
    for (int s = 0; s < b->n; s++) {
        Ctx& c = b->slab[s]->c;
        unsigned stw = 0;
        if (cudaMemcpy(&stw, c.status, sizeof(unsigned), cudaMemcpyDeviceToHost) != cudaSuccess) return PIC_ECUDA;
        if (stw & kErrNan) c.sticky = PIC_ENAN;
        else if (stw & kErrMove) c.sticky = PIC_EMOVE;
        else if (stw & kErrOverflow) c.sticky = PIC_EOVERFLOW;
        if (c.sticky && !b->sticky) b->sticky = c.sticky;
    }
    return b->sticky;
}

int pic_batch_set_timing(pic_batch* b, int32_t enable)
{
    if (!b) return PIC_EINVAL;
    b->timing = enable != 0;
    for (int q = 0; q < 3; q++) b->ms[q] = 0.0;
    for (int q = 0; q < 4; q++) b->nlaunch[q] = 0;
    return PIC_OK;
}

int pic_batch_get_timing(pic_batch* b, double ms[3], int64_t n[4])
{
    if (!b || !ms || !n) return PIC_EINVAL;
    for (int q = 0; q < 3; q++) ms[q] = b->ms[q];
    for (int q = 0; q < 4; q++) n[q] = b->nlaunch[q];
    return PIC_OK;
}

}  // extern "C"
