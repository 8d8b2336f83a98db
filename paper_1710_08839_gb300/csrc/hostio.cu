// Spinor transfer between page-locked host memory and the native device
// layout.
//
// qxd_Dw with page-locked buffers is pipelined over slabs of x0 planes: a
// slab is a contiguous range of the lexicographic host buffer. One stream
// copies the input slabs in (cudaMemcpyAsync, then the pack kernel on the
// device); as soon as slab k is in, D is applied to every output plane whose
// x0 neighbours have arrived (up to the last plane but one of slab k), and
// those planes are unpacked and copied out on a third stream. The two planes
// that wrap around in x0 come last. The copy engines thus use the link in
// both directions at once while the SMs compute, and the output stream
// starts after one input slab. (Kernels reading and writing the host buffers
// directly, in the same pipeline, were 8 % slower: they take SMs from D.)
#include <cstdlib>
#include <new>

#include "dirac_common.cuh"

namespace qxd {

namespace {

// blocks of one layout conversion of the pipeline: it takes part of the GPU
constexpr unsigned kGrid = 152 * 4;

}  // namespace

bool host_device_view(const void* p, void** dev) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();  // clear the error of an unknown pointer
        return false;
    }
    if (a.type != cudaMemoryTypeHost || !a.devicePointer) return false;
    *dev = a.devicePointer;
    return true;
}

// streams (host reads, host writes) and events of the pipeline
constexpr int kMaxSlabs = 16;
struct HostPipe {
    cudaStream_t rd = nullptr, wr = nullptr;
    cudaEvent_t start = nullptr, done = nullptr;
    cudaEvent_t in[kMaxSlabs] = {}, out[kMaxSlabs + 2] = {};
    void* stage_out = nullptr;  // device staging of the lexicographic output
    ~HostPipe() {
        if (stage_out) cudaFree(stage_out);
        if (rd) cudaStreamDestroy(rd);
        if (wr) cudaStreamDestroy(wr);
        cudaEvent_t evs[] = {start, done};
        for (cudaEvent_t e : evs)
            if (e) cudaEventDestroy(e);
        for (cudaEvent_t e : in)
            if (e) cudaEventDestroy(e);
        for (cudaEvent_t e : out)
            if (e) cudaEventDestroy(e);
    }
};

int ensure_hostpipe(qxd_lattice* lat) {
    if (lat->hostpipe) return QXD_OK;
    HostPipe* h = new (std::nothrow) HostPipe();
    if (!h) return fail(QXD_ERR_OOM, "qxd_Dw: host allocation failed");
    lat->hostpipe = h;
    QXD_CUDA(cudaStreamCreateWithFlags(&h->rd, cudaStreamNonBlocking));
    QXD_CUDA(cudaStreamCreateWithFlags(&h->wr, cudaStreamNonBlocking));
    QXD_CUDA(cudaEventCreateWithFlags(&h->start, cudaEventDisableTiming));
    QXD_CUDA(cudaEventCreateWithFlags(&h->done, cudaEventDisableTiming));
    for (cudaEvent_t& e : h->in) QXD_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    for (cudaEvent_t& e : h->out) QXD_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return QXD_OK;
}

// slabs: the largest divisor of N0 up to 16 with at least 2 planes per slab
// (at least 3 slabs, else 0: no pipeline)
int pick_slabs(int N0) {
    int best = 0;
    for (int S = 3; S <= kMaxSlabs; ++S)
        if (N0 % S == 0 && N0 / S >= 2) best = S;
    return best;
}

void release_hostio(qxd_lattice* lat) {
    delete lat->hostpipe;
    lat->hostpipe = nullptr;
}

int dw_host_pipelined(qxd_lattice* lat, void* out_dev, const void* in_dev, int prec, cudaStream_t st) {
    const Geom& g = lat->g;
    const int S = pick_slabs(g.N0);
    if (S < 3) return fail(QXD_ERR_ARG, "qxd_Dw: lattice too short in x0 for the pipelined host path");
    int rc = ensure_hostpipe(lat);
    if (rc) return rc;
    HostPipe& h = *lat->hostpipe;
    const int planes = g.N0 / S;
    const size_t slab = (size_t)planes * g.N1 * g.N2 * g.N3;
    // the pipeline starts after the work already queued on st
    QXD_CUDA(cudaEventRecord(h.start, st));
    QXD_CUDA(cudaStreamWaitEvent(h.rd, h.start, 0));
    QXD_CUDA(cudaStreamWaitEvent(h.wr, h.start, 0));
    const size_t esz = prec == QXD_FP32 ? 24 * sizeof(float) : 24 * sizeof(double);  // bytes per site
    if (!h.stage_out) QXD_CUDA(cudaMalloc(&h.stage_out, (size_t)g.V * 24 * sizeof(double)));
    for (int k = 0; k < S; ++k) {
        QXD_CUDA(cudaMemcpyAsync((char*)lat->scratch_lex + k * slab * esz, (const char*)in_dev + k * slab * esz,
                                 slab * esz, cudaMemcpyDefault, h.rd));
        if ((rc = launch_pack_sites(lat, lat->scratch_in, lat->scratch_lex, prec, k * slab, slab, kGrid, h.rd)))
            return rc;
        QXD_CUDA(cudaEventRecord(h.in[k], h.rd));
    }
    // output planes [lo, hi) once input slab k is in: up to the last plane but
    // one of slab k (its forward neighbour is in slab k + 1); plane 0 (whose
    // backward neighbour is plane N0 - 1) and plane N0 - 1 come last
    const size_t plane = (size_t)g.N1 * g.N2 * g.N3;
    auto out_range = [&](int lo, int hi, int ev) -> int {
        if (hi <= lo) return QXD_OK;
        int r = launch_dirac_planes(lat, lat->scratch_out, lat->scratch_in, prec, lo, hi - lo, st);
        if (r) return r;
        QXD_CUDA(cudaEventRecord(h.out[ev], st));
        QXD_CUDA(cudaStreamWaitEvent(h.wr, h.out[ev], 0));
        if ((r = launch_unpack_sites(lat, h.stage_out, lat->scratch_out, prec, lo * plane, (hi - lo) * plane, kGrid,
                                     h.wr)))
            return r;
        QXD_CUDA(cudaMemcpyAsync((char*)out_dev + lo * plane * esz, (const char*)h.stage_out + lo * plane * esz,
                                 (hi - lo) * plane * esz, cudaMemcpyDefault, h.wr));
        return QXD_OK;
    };
    for (int k = 0; k < S; ++k) {
        QXD_CUDA(cudaStreamWaitEvent(st, h.in[k], 0));  // slabs 0 .. k are in (rd is in order)
        const int lo = k == 0 ? 1 : k * planes - 1;
        const int hi = k == S - 1 ? g.N0 - 1 : (k + 1) * planes - 1;
        if ((rc = out_range(lo, hi, k))) return rc;
    }
    if ((rc = out_range(g.N0 - 1, g.N0, S))) return rc;
    if ((rc = out_range(0, 1, S + 1))) return rc;
    QXD_CUDA(cudaEventRecord(h.done, h.wr));
    QXD_CUDA(cudaStreamWaitEvent(st, h.done, 0));
    return QXD_OK;
}

}  // namespace qxd
