// Host side of the C ABI declared in include/lbm_fs.h: parameter validation,
// device memory, initial upload, step enqueueing (CUDA graphs), read-back.
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <string>
#include <vector>

#include "lbm_fs.h"
#include "lbmfs_handle.h"
#include "lbmfs_internal.h"

using namespace lbmfs;

namespace {
thread_local std::string g_err;
}  // namespace

namespace lbmfs {

lbm_fs_status fail(lbm_fs_status s, const char *fmt, const char *detail) {
    char buf[512];
    snprintf(buf, sizeof buf, fmt, detail ? detail : "");
    g_err = buf;
    return s;
}

lbm_fs_status cuda_fail(cudaError_t e, const char *where) {
    char buf[512];
    snprintf(buf, sizeof buf, "%s: %s", where, cudaGetErrorString(e));
    g_err = buf;
    return e == cudaErrorMemoryAllocation ? LBM_FS_ENOMEM : LBM_FS_ECUDA;
}

lbm_fs_status check_handle(lbm_fs *h) {
    if (!h) return fail(LBM_FS_EINVAL, "null handle%s");
    if (h->dead) return fail(LBM_FS_ESTATE, "handle is in a failed state%s");
    return LBM_FS_OK;
}

#define CK LBMFS_CK

lbm_fs_status read_status(lbm_fs *h) {
    CK(cudaMemcpyAsync(h->pin + lbm_fs::PIN_STATUS, h->d[0].status, sizeof(uint32_t), cudaMemcpyDeviceToHost, h->st));
    CK(cudaStreamSynchronize(h->st));
    uint32_t st;
    memcpy(&st, h->pin + lbm_fs::PIN_STATUS, sizeof st);
    return status_bits(st);
}

lbm_fs_status status_bits(uint32_t st) {
    if (st & ST_OVERFLOW) return fail(LBM_FS_EOVERFLOW, "a device worklist overflowed%s");
    if (st & ST_TIMEOUT) return fail(LBM_FS_ETIMEOUT, "a bounded device wait (staged rows) gave up%s");
    if (st & ST_NONFINITE) return fail(LBM_FS_EUNSTABLE, "non-finite or non-positive density in a fluid cell%s");
    if (st & ST_LIQUID_GAS) return fail(LBM_FS_EUNSTABLE, "a liquid cell touched a gas cell (open interface layer)%s");
    if (st & ST_CONTACT) return fail(LBM_FS_EUNSTABLE, "a moving body reached a domain wall (body-wall contact is not modelled)%s");
    if (st & ST_TOP) return fail(LBM_FS_EUNSTABLE, "fluid appeared above the bulk kernel's tracked fluid top%s");
    return LBM_FS_OK;
}

cudaError_t Sides::create() {
    int lo = 0, hi = 0;
    cudaError_t e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
    for (int k = 0; k < SIDE_STREAMS && e == cudaSuccess; ++k) {
        e = cudaStreamCreateWithPriority(&st[k], cudaStreamNonBlocking, hi);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join[k], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork2, cudaEventDisableTiming);
    return e;
}
void Sides::destroy() {
    for (int k = 0; k < SIDE_STREAMS; ++k) {
        if (st[k]) cudaStreamDestroy(st[k]);
        if (join[k]) cudaEventDestroy(join[k]);
        st[k] = nullptr;
        join[k] = nullptr;
    }
    if (fork) cudaEventDestroy(fork);
    if (fork2) cudaEventDestroy(fork2);
    fork = fork2 = nullptr;
}

void begin_mass(lbm_fs *h) {
    if (h->started) return;
    h->ks.liquid_mass(h->d[h->cur], h->st);
    cudaMemcpyAsync(h->d[0].ledger + LG_MASS0, h->d[0].ledger + LG_MASS, sizeof(double), cudaMemcpyDeviceToDevice,
                    h->st);
    h->started = true;
}

}  // namespace lbmfs

namespace {

lbm_fs_status capture_graphs(lbm_fs *h) {
    for (int k = 0; k < 2; ++k) {
        if (h->gexec[k]) {
            cudaGraphExecDestroy(h->gexec[k]);
            h->gexec[k] = nullptr;
        }
    }
    for (int k = 0; k < 2; ++k) {
        cudaGraph_t g = nullptr;
        CK(cudaStreamBeginCapture(h->cap_st, cudaStreamCaptureModeThreadLocal));
        h->per_step = h->ks.step(h->d[k], h->cap_st, &h->sides, nullptr);
        cudaError_t e = cudaStreamEndCapture(h->cap_st, &g);
        if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
        e = cudaGraphInstantiate(&h->gexec[k], g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
    }
    h->graph_nb = h->nb;
    return LBM_FS_OK;
}

void set_grids(lbm_fs *h, void *fA, void *fB, double *pA, double *pB) {
    h->d[0].fsrc = fA;
    h->d[0].fdst = fB;
    h->d[0].phisrc = pA;
    h->d[0].phidst = pB;
    h->d[1].fsrc = fB;
    h->d[1].fdst = fA;
    h->d[1].phisrc = pB;
    h->d[1].phidst = pA;
}

size_t storage_bytes(int storage, long long N) {
    switch (storage) {
        case LBM_FS_F64: return (size_t)N * Q * 8;
        case LBM_FS_F32: return (size_t)N * Q * 4;
        default: return (size_t)N * (4 + (Q - 1) * 2);
    }
}

}  // namespace

extern "C" {

int32_t lbm_fs_version(void) { return 1; }

const char *lbm_fs_last_error_string(void) { return g_err.c_str(); }

lbm_fs_status lbm_fs_create(const lbm_fs_params *p, lbm_fs **out) {
    if (!p || !out) return fail(LBM_FS_EINVAL, "null argument%s");
    *out = nullptr;
    if (p->nx <= 0 || p->ny <= 0 || p->nz <= 0) return fail(LBM_FS_EINVAL, "grid sizes must be positive%s");
    long long N = (long long)p->nx * p->ny * p->nz;
    if (N >= 0xFFFFFFFFll) return fail(LBM_FS_EINVAL, "grid has 2^32 cells or more%s");
    // the float storages' bulk kernel indexes a population as q N + cell in 32 bits
    if (p->storage != LBM_FS_F64 && N * Q >= 0xFFFFFFFFll)
        return fail(LBM_FS_EINVAL, "float storages take fewer than 2^32 / 19 cells%s");
    if (!(p->tau > 0.5) || !std::isfinite(p->tau)) return fail(LBM_FS_EINVAL, "tau must exceed 1/2%s");
    if (p->storage < LBM_FS_F64 || p->storage > LBM_FS_F16S) return fail(LBM_FS_EINVAL, "unknown storage%s");
    if (!p->init_flags || !p->init_fill || !p->init_rho) return fail(LBM_FS_EINVAL, "init_flags, init_fill and init_rho are required%s");
    if (!(p->rho_gas > 0.0) || !(p->eps >= 0.0)) return fail(LBM_FS_EINVAL, "rho_gas must be positive and eps non-negative%s");
    if ((p->dev_alloc == nullptr) != (p->dev_free == nullptr)) return fail(LBM_FS_EINVAL, "dev_alloc and dev_free go together%s");
    if (!(p->sigma >= 0.0) || !std::isfinite(p->sigma)) return fail(LBM_FS_EINVAL, "sigma must be finite and >= 0%s");
    for (int f = 0; f < 6; ++f)
        for (int k = 0; k < 3; ++k)
            if (!std::isfinite(p->wall_vel[f][k])) return fail(LBM_FS_EINVAL, "non-finite wall velocity%s");
    const bool rd_db = p->readings & LBM_FS_READING_DEADBAND, rd_vm = p->readings & LBM_FS_READING_VIRTUAL_MASS;
    if (rd_db && !(p->normal_deadband >= 0.0 && std::isfinite(p->normal_deadband)))
        return fail(LBM_FS_EINVAL, "normal_deadband must be finite and >= 0%s");
    if (rd_vm && !(p->virtual_mass >= 0.0 && std::isfinite(p->virtual_mass)))
        return fail(LBM_FS_EINVAL, "virtual_mass must be finite and >= 0%s");
    double proj = 0.0;
    for (int k = 0; k < 3; ++k) {
        double a = fabs(p->gravity[k] + p->body_accel[k]);
        if (!std::isfinite(a)) return fail(LBM_FS_EINVAL, "non-finite acceleration%s");
        proj += a * (k == 0 ? p->nx : (k == 1 ? p->ny : p->nz));
    }
    // Sec. 2.1 incompressibility condition (l_x, l_y, l_z) . a << c_s^2 = 1/3
    if (proj >= 1.0 / 3.0) return fail(LBM_FS_EINVAL, "(nx, ny, nz) . |a| must stay well below c_s^2 = 1/3%s");

    lbm_fs *h = new lbm_fs();
    h->p = *p;
    h->p.init_flags = nullptr;
    h->p.init_fill = nullptr;
    h->p.init_rho = nullptr;
    h->p.init_vel = nullptr;
    h->st = (cudaStream_t)p->stream;
    switch (p->storage) {
        case LBM_FS_F64: h->ks = kernels_f64(); break;
        case LBM_FS_F32: h->ks = kernels_f32(); break;
        default: h->ks = kernels_f16s(); break;
    }
    auto bail = [&](lbm_fs_status s) {
        h->release();
        delete h;
        return s;
    };
    cudaError_t e = cudaStreamCreateWithFlags(&h->cap_st, cudaStreamNonBlocking);
    if (e == cudaSuccess && p->use_graphs) e = h->sides.create();
    if (e == cudaSuccess) e = cudaHostAlloc((void **)&h->pin, lbm_fs::PIN_BYTES, cudaHostAllocDefault);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaStreamCreate"));

    Dev d{};
    d.nx = p->nx;
    d.ny = p->ny;
    d.nz = p->nz;
    d.periodic = p->periodic & 7u;
    d.N = N;
    d.omega = 1.0 / p->tau;
    for (int k = 0; k < 3; ++k) {
        d.a[k] = p->gravity[k] + p->body_accel[k];
        d.grav[k] = p->gravity[k];
    }
    d.rho_g = p->rho_gas;
    d.eps = p->eps;
    d.omega_f = (float)d.omega;
    for (int k = 0; k < 3; ++k) d.a_f[k] = (float)d.a[k];
    d.drg_f = (float)(d.rho_g - 1.0);
    d.rg1_f = (float)(1.0 - d.rho_g);
    d.sigma = p->sigma;
    d.sigma_f = (float)p->sigma;
    d.cap = (uint32_t)N;
    d.deadband = rd_db ? p->normal_deadband : 1e-2;
    d.deadband_f = (float)d.deadband;
    d.vmass = rd_vm ? p->virtual_mass : 1.0;
    d.force_mean = (p->readings & LBM_FS_READING_FORCE_MEAN) ? (p->force_mean != 0) : 1;
    d.nb_rule = (p->readings & LBM_FS_READING_NEIGHBOUR_RULE) ? (p->neighbour_rule != 0) : 1;
    d.pair_ok = p->nx % 2 == 0 && N % 2 == 0;
    // bulk-kernel variant (float storages): LBMFS_BULK=pipe|tma selects the staged
    // variants instead of the default (both measured slower on GB300; the TMA one
    // needs rows of 16-byte multiples)
    d.bulk = BULK_PLAIN;
    if (const char *v = getenv("LBMFS_BULK")) {
        if (!strcmp(v, "pipe")) d.bulk = BULK_PIPE;
        else if (!strcmp(v, "tma")) d.bulk = BULK_TMA;
    }
    if (d.bulk == BULK_TMA &&
        !((p->storage == LBM_FS_F32 && p->nx % 4 == 0) || (p->storage == LBM_FS_F16S && p->nx % 8 == 0)))
        d.bulk = BULK_PLAIN;
    size_t fb = storage_bytes(p->storage, N);
    size_t nb4 = ((size_t)N + 3) & ~(size_t)3;
    // (the ring kernel reads the class bytes of whole tiles: zeros after the grid)
    const size_t nflags = ((size_t)N + RING_TILE - 1) / RING_TILE * RING_TILE;
    d.flags = (uint8_t *)h->alloc(nflags);
    d.bid = (uint8_t *)h->alloc(nb4);
    d.cmark = (uint8_t *)h->alloc(nb4);
    // population grids with guard bands: the staged bulk kernel reads a
    // 16-byte halo around each row segment, which at the grid's
    // first and last rows reaches past the population array; the ring kernel's
    // tiles reach a z-plane, a row and a tile further (multiples of 16 bytes)
    size_t guard = GRID_GUARD;
    if (p->storage == LBM_FS_F16S) guard += (((size_t)p->nx * p->ny + p->nx + 1024) * 2 + 255) & ~(size_t)255;
    void *fA = h->alloc(fb + 2 * guard), *fB = h->alloc(fb + 2 * guard);
    if (fA) fA = (char *)fA + guard;
    if (fB) fB = (char *)fB + guard;
    double *pA = (double *)h->alloc(N * 8), *pB = (double *)h->alloc(N * 8);
    d.m = (double *)h->alloc(N * 8);
    for (int k : {WL_FILLED, WL_EMPTIED, WL_COVER}) d.list[k] = (uint32_t *)h->alloc(N * 4);
    // what a step reads of the one before it, in turn: the lists prev_wl(k), the
    // counters and the body records
    uint32_t *lists[2];
    for (auto &l : lists) l = (uint32_t *)h->alloc((size_t)N * 4 * PREV_LISTS);
    d.cnt = (uint32_t *)h->alloc(2 * CN_COUNT * 4);
    d.bodies = (Body *)h->alloc(2 * sizeof(Body) * MAX_BODIES);
    const size_t pfb = p->storage == LBM_FS_F64 ? 0 : (size_t)N * 4;
    float *pfA = (float *)h->alloc(pfb), *pfB = (float *)h->alloc(pfb);
    d.part = (double *)h->alloc(2 * sizeof(double) * MAX_BODIES * FORCE_BLOCKS * 7);
    d.part128 = p->storage == LBM_FS_F64;
    d.range_blocks = FORCE_BLOCKS;
    d.ledger = (double *)h->alloc(sizeof(double) * LG_COUNT);
    d.status = (uint32_t *)h->alloc(16);
    d.red = (double *)h->alloc(sizeof(double) * LIST_BLOCKS);
    double *wallv = (double *)h->alloc(sizeof(double) * 18);
    d.wallv = wallv;
    int *ztop = (int *)h->alloc(sizeof(int) * 2);
    for (void *ptr : h->allocs)
        if (!ptr) return bail(fail(LBM_FS_ENOMEM, "device allocation failed%s"));
    if (h->allocs.size() != 23) return bail(fail(LBM_FS_ENOMEM, "device allocation failed%s"));
    if (h->misaligned) return bail(fail(LBM_FS_EINVAL, "dev_alloc must return 16-byte aligned memory%s"));
    d.walls_move = 0;
    for (int f = 0; f < 6; ++f)
        for (int k = 0; k < 3; ++k)
            if (p->wall_vel[f][k] != 0.0 && !(d.periodic & (1u << (f / 2)))) d.walls_move = 1;
    cudaStream_t st = h->st;
#define CKB(call)                                                   \
    do {                                                            \
        cudaError_t e_ = (call);                                    \
        if (e_ != cudaSuccess) return bail(cuda_fail(e_, #call));   \
    } while (0)
    CKB(cudaMemsetAsync(d.cmark, 0, nb4, st));
    CKB(cudaMemsetAsync(d.flags, 0, nflags, st));
    CKB(cudaMemsetAsync((char *)fA - guard, 0, fb + 2 * guard, st));
    CKB(cudaMemsetAsync((char *)fB - guard, 0, fb + 2 * guard, st));
    CKB(cudaMemsetAsync(pA, 0, N * 8, st));
    CKB(cudaMemsetAsync(pB, 0, N * 8, st));
    CKB(cudaMemsetAsync(d.m, 0, N * 8, st));
    CKB(cudaMemsetAsync(pfA, 0, pfb, st));
    CKB(cudaMemsetAsync(pfB, 0, pfb, st));
    CKB(cudaMemsetAsync(d.cnt, 0, 2 * CN_COUNT * 4, st));
    CKB(cudaMemsetAsync(d.bodies, 0, 2 * sizeof(Body) * MAX_BODIES, st));
    CKB(cudaMemsetAsync(d.ledger, 0, sizeof(double) * LG_COUNT, st));
    CKB(cudaMemsetAsync(d.status, 0, 16, st));
    CKB(cudaMemsetAsync(d.part, 0, 2 * sizeof(double) * MAX_BODIES * FORCE_BLOCKS * 7, st));
    CKB(cudaMemcpyAsync(wallv, &p->wall_vel[0][0], sizeof(double) * 18, cudaMemcpyHostToDevice, st));
    // the first step visits every tile (its read slot: nz) and records the top
    const int zt0[2] = {p->nz, -1};
    CKB(cudaMemcpyAsync(ztop, zt0, sizeof zt0, cudaMemcpyHostToDevice, st));
    h->d[0] = d;
    h->d[1] = d;
    set_grids(h, fA, fB, pA, pB);
    for (int k = 0; k < 2; ++k) {
        Dev &e = h->d[k];
        e.phifsrc = k ? pfB : pfA;
        e.phifdst = k ? pfA : pfB;
        e.bodies = d.bodies + k * MAX_BODIES;
        e.bodies_new = d.bodies + (k ^ 1) * MAX_BODIES;
        e.cnt = d.cnt + k * CN_COUNT;
        e.pcnt = d.cnt + (k ^ 1) * CN_COUNT;
        for (int j = 0; j < PREV_LISTS; ++j) {
            e.list[prev_wl(j)] = lists[k] + (size_t)N * j;
            e.plist[j] = lists[k ^ 1] + (size_t)N * j;
        }
        // What the conversions and the remap need for themselves lies in arrays
        // that the step has read by then: its previous step's lists (by the
        // interface kernel; next written by the next step) and its source fill
        // levels (by the force and interface kernels).  With them on their own
        // a cell took 21 bytes more.
        static_assert(PREV_LISTS == 4, "an entry's 16 bytes: rphi 8, receivers 4, rdec 1");
        uint32_t *spent = lists[k ^ 1];
        e.rphi = (double *)spent;
        e.list[WL_RECV] = spent + (size_t)N * 2;
        e.rdec = (uint8_t *)(spent + (size_t)N * 3);
        e.rrho = e.phisrc;
    }
    h->d[0].ztop_rd = ztop;
    h->d[0].ztop_wr = ztop + 1;
    h->d[1].ztop_rd = ztop + 1;
    h->d[1].ztop_wr = ztop;

    // upload the initial state (staged through temporary device buffers)
    const uint8_t *dfl = p->init_flags;
    const double *dfi = p->init_fill, *drh = p->init_rho, *dvl = p->init_vel;
    void *tmp = nullptr;
    if (!p->init_on_device) {
        size_t bytes = (size_t)N * (1 + 8 + 8) + (p->init_vel ? (size_t)N * 24 : 0) + 64;
        CKB(cudaMalloc(&tmp, bytes));
        char *c = (char *)tmp;
        double *tfi = (double *)c;
        double *trh = tfi + N;
        double *tvl = p->init_vel ? trh + N : nullptr;
        uint8_t *tfl = (uint8_t *)(p->init_vel ? tvl + 3 * N : trh + N);
        CKB(cudaMemcpyAsync(tfl, p->init_flags, N, cudaMemcpyHostToDevice, st));
        CKB(cudaMemcpyAsync(tfi, p->init_fill, N * 8, cudaMemcpyHostToDevice, st));
        CKB(cudaMemcpyAsync(trh, p->init_rho, N * 8, cudaMemcpyHostToDevice, st));
        if (tvl) CKB(cudaMemcpyAsync(tvl, p->init_vel, N * 24, cudaMemcpyHostToDevice, st));
        dfl = tfl;
        dfi = tfi;
        drh = trh;
        dvl = tvl;
    }
    h->ks.init_cells(h->d[0], dfl, dfi, drh, dvl, st);
    e = cudaGetLastError();
    uint32_t loose = 0;  // obstacles among the initial classes
    if (e == cudaSuccess) e = cudaMemcpyAsync(&loose, d.status + 3, sizeof loose, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (tmp) cudaFree(tmp);
    if (e != cudaSuccess) return bail(cuda_fail(e, "initial upload"));
    h->d[0].loose = h->d[1].loose = loose != 0;
#undef CKB
    *out = h;
    return LBM_FS_OK;
}

lbm_fs_status lbm_fs_destroy(lbm_fs *h) {
    if (!h) return fail(LBM_FS_EINVAL, "null handle%s");
    if (h->owner) return fail(LBM_FS_ESTATE, "the tank belongs to a batch (lbm_fs_batch_destroy frees it)%s");
    cudaStreamSynchronize(h->st);
    h->release();
    delete h;
    return LBM_FS_OK;
}

lbm_fs_status lbm_fs_add_box(lbm_fs *h, const lbm_fs_box *b, int32_t *out_id) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    if (!b) return fail(LBM_FS_EINVAL, "null box%s");
    if (h->nb >= MAX_BODIES) return fail(LBM_FS_EINVAL, "at most 255 boxes%s");
    for (int k = 0; k < 3; ++k)
        if (!(b->half[k] > 0.0) || !std::isfinite(b->center[k])) return fail(LBM_FS_EINVAL, "box half extents must be positive%s");
    double qn = std::sqrt(b->quat[0] * b->quat[0] + b->quat[1] * b->quat[1] + b->quat[2] * b->quat[2] + b->quat[3] * b->quat[3]);
    if (!(qn > 0.5 && qn < 2.0)) return fail(LBM_FS_EINVAL, "quaternion must be (close to) unit%s");
    if (!(b->density_ratio > 0.0)) return fail(LBM_FS_EINVAL, "density_ratio must be positive%s");
    int base = b->mode & 0xff;
    if (base > 2 || (b->mode & ~0x1ff)) return fail(LBM_FS_EINVAL, "unknown mode%s");
    if (b->shape != 0 && b->shape != 1) return fail(LBM_FS_EINVAL, "unknown shape%s");
    Body hb;
    memset(&hb, 0, sizeof hb);
    for (int k = 0; k < 3; ++k) {
        hb.o[k] = b->center[k];
        hb.h[k] = b->half[k];
        hb.v[k] = b->vel[k];
        hb.w[k] = b->omega[k];
        hb.axis[k] = b->rot_axis[k];
    }
    for (int k = 0; k < 4; ++k) hb.q[k] = b->quat[k];
    hb.dens = b->density_ratio;
    hb.damp = b->lin_damping;
    hb.mode = b->mode;
    hb.shape = b->shape;
    int id = h->nb;
    // the cells of its range, for the launches that look through it
    double range = 1.0;
    const double *q = b->quat, R[9] = {1 - 2 * (q[2] * q[2] + q[3] * q[3]), 2 * (q[1] * q[2] - q[0] * q[3]), 2 * (q[1] * q[3] + q[0] * q[2]),
                                       2 * (q[1] * q[2] + q[0] * q[3]), 1 - 2 * (q[1] * q[1] + q[3] * q[3]), 2 * (q[2] * q[3] - q[0] * q[1]),
                                       2 * (q[1] * q[3] - q[0] * q[2]), 2 * (q[2] * q[3] + q[0] * q[1]), 1 - 2 * (q[1] * q[1] + q[2] * q[2])};
    const int n3[3] = {h->p.nx, h->p.ny, h->p.nz};
    for (int k = 0; k < 3; ++k) {
        double e = b->half[0];
        if (b->shape == 0) e = fabs(R[3 * k]) * b->half[0] + fabs(R[3 * k + 1]) * b->half[1] + fabs(R[3 * k + 2]) * b->half[2];
        range *= std::min(2.0 * e + 5.0, (double)n3[k]);
    }
    const int blocks = (int)std::min<double>(range / RANGE_CELLS, RANGE_BLOCKS_MAX);
    cudaStream_t st = h->st;
    CK(cudaMemcpyAsync(h->d[h->cur].bodies + id, &hb, sizeof hb, cudaMemcpyHostToDevice, st));
    CK(cudaStreamSynchronize(st));
    h->nb++;
    for (int k = 0; k < 2; ++k) {
        h->d[k].nb = h->nb;
        h->d[k].range_blocks = std::max(h->d[k].range_blocks, blocks);
    }
    h->ks.body_prepare(h->d[h->cur], id, st);
    h->ks.map_body(h->d[h->cur], id, h->started ? 1 : 0, st);
    CK(cudaGetLastError());
    if (out_id) *out_id = id;
    return LBM_FS_OK;
}

lbm_fs_status lbm_fs_step(lbm_fs *h, int32_t nsteps) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    if (h->owner) return fail(LBM_FS_ESTATE, "the tank belongs to a batch (step it with lbm_fs_batch_step)%s");
    if (nsteps < 0) return fail(LBM_FS_EINVAL, "nsteps must be >= 0%s");
    if (nsteps == 0) return LBM_FS_OK;
    cudaStream_t st = h->st;
    begin_mass(h);
    CK(cudaGetLastError());
    if (h->p.use_graphs && h->graph_nb != h->nb) {
        s = capture_graphs(h);
        if (s) return s;
    }
    for (int32_t k = 0; k < nsteps; ++k) {
        if (h->p.use_graphs) {
            CK(cudaGraphLaunch(h->gexec[h->cur], st));
        } else {
            h->per_step = h->ks.step(h->d[h->cur], st, nullptr, nullptr);
            CK(cudaGetLastError());
        }
        h->launches += h->per_step;
        h->cur ^= 1;
        h->step++;
    }
    return LBM_FS_OK;
}

lbm_fs_status lbm_fs_sync(lbm_fs *h) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    return read_status(h);
}

lbm_fs_status lbm_fs_body_state(lbm_fs *h, int32_t id, lbm_fs_body_state_t *out) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    if (id < 0 || id >= h->nb || !out) return fail(LBM_FS_EINVAL, "bad body id%s");
    return lbm_fs_body_states(h, id, 1, out);
}

lbm_fs_status lbm_fs_body_states(lbm_fs *h, int32_t first, int32_t count, lbm_fs_body_state_t *out) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    if (first < 0 || count < 0 || first + count > h->nb || (count > 0 && !out))
        return fail(LBM_FS_EINVAL, "bad body range%s");
    if (count == 0) return read_status(h);
    // the status word comes with the bodies: one synchronisation
    const size_t bytes = sizeof(Body) * (size_t)count;
    std::vector<Body> many;
    Body *hb = reinterpret_cast<Body *>(h->pin + lbm_fs::PIN_DATA);
    if (bytes > lbm_fs::PIN_BYTES - lbm_fs::PIN_DATA) {
        many.resize(count);
        hb = many.data();
    }
    CK(cudaMemcpyAsync(hb, h->d[h->cur].bodies + first, bytes, cudaMemcpyDeviceToHost, h->st));
    const lbm_fs_status s1 = read_status(h);
    if (s1 == LBM_FS_ECUDA || s1 == LBM_FS_ENOMEM) return s1;
    for (int32_t b = 0; b < count; ++b) {
        for (int k = 0; k < 3; ++k) {
            out[b].F[k] = hb[b].F[k];
            out[b].T[k] = hb[b].T[k];
            out[b].center[k] = hb[b].o[k];
            out[b].vel[k] = hb[b].v[k];
            out[b].omega[k] = hb[b].w[k];
        }
        for (int k = 0; k < 4; ++k) out[b].quat[k] = hb[b].q[k];
        out[b].S = hb[b].S;
    }
    return s1;
}

lbm_fs_status lbm_fs_forces(lbm_fs *h, int32_t id, double F[3], double T[3], double center[3], double quat[4]) {
    lbm_fs_body_state_t bs;
    lbm_fs_status s = lbm_fs_body_state(h, id, &bs);
    if (s != LBM_FS_OK && s != LBM_FS_EUNSTABLE && s != LBM_FS_EOVERFLOW) return s;
    for (int k = 0; k < 3; ++k) {
        if (F) F[k] = bs.F[k];
        if (T) T[k] = bs.T[k];
        if (center) center[k] = bs.center[k];
    }
    if (quat)
        for (int k = 0; k < 4; ++k) quat[k] = bs.quat[k];
    return s;
}

lbm_fs_status lbm_fs_read_fields(lbm_fs *h, uint32_t mask, void *const *dst, int32_t dst_on_device) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    if (!dst || (mask & ~63u)) return fail(LBM_FS_EINVAL, "bad field mask or destination%s");
    for (int k = 0; k < 6; ++k)
        if ((mask & (1u << k)) && !dst[k]) return fail(LBM_FS_EINVAL, "missing destination buffer%s");
    const long long N = h->d[0].N;
    const size_t sz[6] = {(size_t)N, (size_t)N * 8, (size_t)N * 8, (size_t)N * 8, (size_t)N * 24, (size_t)N * 8 * Q};
    cudaStream_t st = h->st;
    void *ddst[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    std::vector<void *> tmp;
    for (int k = 0; k < 6; ++k) {
        if (!(mask & (1u << k))) continue;
        if (dst_on_device) {
            ddst[k] = dst[k];
        } else {
            void *ptr = nullptr;
            cudaError_t e = cudaMalloc(&ptr, sz[k]);
            if (e != cudaSuccess) {
                for (void *t : tmp) cudaFree(t);
                return cuda_fail(e, "read_fields staging");
            }
            tmp.push_back(ptr);
            ddst[k] = ptr;
        }
    }
    h->ks.read_fields(h->d[h->cur], mask, ddst, st);
    cudaError_t e = cudaGetLastError();
    for (int k = 0; k < 6 && e == cudaSuccess; ++k)
        if (!dst_on_device && (mask & (1u << k))) e = cudaMemcpyAsync(dst[k], ddst[k], sz[k], cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && tmp.empty()) return read_status(h);  // (waits for the fields too)
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    for (void *t : tmp) cudaFree(t);
    if (e != cudaSuccess) return cuda_fail(e, "read_fields");
    return read_status(h);
}

lbm_fs_status lbm_fs_stats(lbm_fs *h, lbm_fs_stats_t *out) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    if (!out) return fail(LBM_FS_EINVAL, "null output%s");
    cudaStream_t st = h->st;
    h->ks.liquid_mass(h->d[h->cur], st);
    CK(cudaGetLastError());
    double lg[LG_COUNT];
    uint32_t cnt[CN_COUNT], status;
    static_assert(lbm_fs::PIN_DATA + sizeof lg + sizeof cnt <= lbm_fs::PIN_BYTES, "the statistics fit the pinned buffer");
    char *plg = h->pin + lbm_fs::PIN_DATA, *pcnt = plg + sizeof lg;
    CK(cudaMemcpyAsync(plg, h->d[0].ledger, sizeof lg, cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(pcnt, h->d[h->cur ^ 1].cnt, sizeof cnt, cudaMemcpyDeviceToHost, st));  // of the last step
    const lbm_fs_status s1 = read_status(h);
    if (s1 == LBM_FS_ECUDA || s1 == LBM_FS_ENOMEM) return s1;
    memcpy(lg, plg, sizeof lg);
    memcpy(cnt, pcnt, sizeof cnt);
    if (h->step == 0) memset(cnt, 0, sizeof cnt);
    memcpy(&status, h->pin + lbm_fs::PIN_STATUS, sizeof status);
    memset(out, 0, sizeof *out);
    out->step = h->step;
    out->liquid_mass = lg[LG_MASS];
    out->mass0 = h->started ? lg[LG_MASS0] : lg[LG_MASS];
    out->covered = lg[LG_COVERED];
    out->uncovered = lg[LG_UNCOVERED];
    out->lost_excess = lg[LG_LOST];
    out->n_interface = cnt[WL_IFACE];
    out->n_filled = cnt[WL_FILLED];
    out->n_emptied = cnt[WL_EMPTIED];
    out->n_new_from_gas = cnt[WL_NEWG];
    out->n_new_from_liquid = cnt[WL_NEWL];
    out->n_pending = cnt[WL_PEND];
    out->status = status;
    out->kernel_launches = h->launches;
    out->wall_source = lg[LG_WALL];
    out->n_general = cnt[CN_NEAR];
    return s1;
}

lbm_fs_status lbm_fs_kernel_times(lbm_fs *h, int32_t nsteps, double *ms, const char **names, int32_t cap, int32_t *nk) {
    lbm_fs_status s = check_handle(h);
    if (s) return s;
    if (h->owner) return fail(LBM_FS_ESTATE, "the tank belongs to a batch (use lbm_fs_batch_kernel_times)%s");
    if (nsteps <= 0 || !ms || cap <= 0) return fail(LBM_FS_EINVAL, "bad arguments%s");
    const int K = h->ks.nkernels;
    std::vector<cudaEvent_t> ev(K + 1);
    for (auto &x : ev) CK(cudaEventCreate(&x));
    std::vector<double> acc(K, 0.0);
    cudaStream_t st = h->st;
    begin_mass(h);
    CK(cudaGetLastError());
    for (int32_t it = 0; it < nsteps; ++it) {
        int n = h->ks.step(h->d[h->cur], st, nullptr, ev.data());
        CK(cudaGetLastError());
        CK(cudaEventSynchronize(ev[K]));
        for (int k = 0; k < K; ++k) {
            float t = 0.0f;
            CK(cudaEventElapsedTime(&t, ev[k], ev[k + 1]));
            acc[k] += t;
        }
        h->launches += n;
        h->cur ^= 1;
        h->step++;
    }
    for (auto &x : ev) cudaEventDestroy(x);
    int m = K < cap ? K : cap;
    for (int k = 0; k < m; ++k) {
        ms[k] = acc[k];
        if (names) names[k] = h->ks.names[k];
    }
    if (nk) *nk = K;
    return read_status(h);
}

}  // extern "C"
