// claw_hostloop.cu -- stepping a level whose state lives in host memory (claw_steps_from_host): the
// level is taken in pieces of boxes, each copied in, stepped and copied back on streams of its own
// kind, so that the copies of both directions and the steps overlap.
//
// The loop enqueues about fifteen calls a piece and step.  From Python that took some 100 us a piece
// and step, which bound every level below 60 MB (1024^2 in eight pieces: 794 us a step); here it takes
// 13 us (1024^2: 221 us in four pieces, 25 MB each way).
#include "claw_host.h"

using namespace claw_host;

namespace {

struct Failed {
    cudaError_t e = cudaSuccess;
    int rc = CLAW_OK;
    void operator()(cudaError_t x)
    {
        if (e == cudaSuccess) e = x;
    }
    void status(int x)
    {
        if (rc == CLAW_OK) rc = x;
    }
    bool any() const { return e != cudaSuccess || rc != CLAW_OK; }
};

// the streams and events of a context's host-resident loop (kept from call to call)
int ensure_loop(claw_ctx* ctx, int pieces)
{
    HostLoop& h = ctx->hostloop;
    for (cudaStream_t& s : h.streams)
        if (!s && cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return CLAW_ECUDA;
    const size_t want = (size_t)HostLoop::kinds * pieces + 1;
    while (h.events.size() < want) {
        cudaEvent_t e;
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return CLAW_ENOMEM;
        h.events.push_back(e);
    }
    return CLAW_OK;
}

}  // namespace

extern "C" int claw_steps_from_host(claw_ctx* ctx, double* q0, double* q1, const double* aux, double* dt, double* smax,
                                    double* host_a, double* host_b, double* stage_in, double* stage_out,
                                    int32_t nsteps, int32_t npieces, const int32_t* piece_boxes,
                                    const int64_t* ranges, const int32_t* need_start, const int32_t* needs,
                                    void* stream)
{
    if (!valid_level(ctx, 0) || !q0 || !q1 || !dt || !smax || !host_a || !host_b || nsteps < 0 || npieces < 1 ||
        !piece_boxes || !ranges || !need_start || !needs || (stage_in == nullptr) != (stage_out == nullptr))
        return CLAW_EINVAL;
    // a packed buffer holds the level's packed interiors; how far a pool reaches only the caller knows
    const int64_t most = stage_in ? (int64_t)ctx->lev[0].packed : INT64_MAX / (int64_t)sizeof(double);
    for (int k = 0; k < npieces; ++k) {
        if (piece_boxes[k] < 0 || piece_boxes[k + 1] < piece_boxes[k] || piece_boxes[k + 1] > ctx->lev[0].nboxes ||
            ranges[2 * k] < 0 || ranges[2 * k + 1] < ranges[2 * k] || ranges[2 * k + 1] > most || need_start[k] < 0 ||
            need_start[k + 1] < need_start[k])
            return CLAW_EINVAL;
        for (int m = need_start[k]; m < need_start[k + 1]; ++m)
            if (needs[m] < 0 || needs[m] >= npieces) return CLAW_EINVAL;
    }
    if (nsteps == 0) return CLAW_OK;
    DevGuard g(ctx->device);
    if (int rc = ensure_loop(ctx, npieces)) return rc;
    HostLoop& h = ctx->hostloop;
    cudaStream_t comp = (cudaStream_t)stream, s_in = h.streams[0], s_out = h.streams[1], s_un = h.streams[2],
                 s_pk = h.streams[3];
    // per piece: its copy has landed, it is in the pool, it is stepped, packed, back on the host
    auto ev = [&](int kind, int k) { return h.events[(size_t)kind * npieces + k + 1]; };
    enum { LANDED, ARRIVED, STEPPED, PACKED, LEFT };
    static_assert(HostLoop::kinds == LEFT + 1, "an event per kind and piece");
    const bool packed = stage_in != nullptr;
    Failed f;
    f(cudaEventRecord(h.events[0], comp));
    for (cudaStream_t s : h.streams) f(cudaStreamWaitEvent(s, h.events[0], 0));
    double *src = host_a, *dst = host_b, *q = q0, *qn = q1;
    for (int n = 0; n < nsteps && !f.any(); ++n) {
        for (int k = 0; k < npieces; ++k) {
            const int64_t a = ranges[2 * k], bytes = (ranges[2 * k + 1] - a) * (int64_t)sizeof(double);
            if (n) f(cudaStreamWaitEvent(s_in, ev(LEFT, k), 0));   // this piece of the previous step is on the host
            if (packed) {
                if (n) f(cudaStreamWaitEvent(s_in, ev(ARRIVED, k), 0));   // its staging slot has been read
                f(cudaMemcpyAsync(stage_in + a, src + a, bytes, cudaMemcpyDefault, s_in));
                f(cudaEventRecord(ev(LANDED, k), s_in));
                f(cudaStreamWaitEvent(s_un, ev(LANDED, k), 0));
                f.status(claw_unpack_interiors(ctx, 0, piece_boxes[k], piece_boxes[k + 1], stage_in, q, s_un));
                f(cudaEventRecord(ev(ARRIVED, k), s_un));
            } else {
                f(cudaMemcpyAsync(q + a, src + a, bytes, cudaMemcpyDefault, s_in));
                f(cudaEventRecord(ev(ARRIVED, k), s_in));
            }
        }
        for (int k = 0; k < npieces; ++k) {
            for (int m = need_start[k]; m < need_start[k + 1]; ++m)
                f(cudaStreamWaitEvent(comp, ev(ARRIVED, needs[m]), 0));
            f.status(claw_level_advance_boxes(ctx, 0, piece_boxes[k], piece_boxes[k + 1], q, qn, aux, dt, smax,
                                              CLAW_ADVANCE_PULL_GHOSTS, comp));
            f(cudaEventRecord(ev(STEPPED, k), comp));
        }
        f.status(claw_dt_update(ctx, 0, smax, dt, comp));
        for (int k = 0; k < npieces; ++k) {
            const int64_t a = ranges[2 * k], bytes = (ranges[2 * k + 1] - a) * (int64_t)sizeof(double);
            if (packed) {
                f(cudaStreamWaitEvent(s_pk, ev(STEPPED, k), 0));
                if (n) f(cudaStreamWaitEvent(s_pk, ev(LEFT, k), 0));   // its out staging slot has been copied out
                f.status(claw_pack_interiors(ctx, 0, piece_boxes[k], piece_boxes[k + 1], qn, stage_out, s_pk));
                f(cudaEventRecord(ev(PACKED, k), s_pk));
                f(cudaStreamWaitEvent(s_out, ev(PACKED, k), 0));
                f(cudaMemcpyAsync(dst + a, stage_out + a, bytes, cudaMemcpyDefault, s_out));
            } else {
                f(cudaStreamWaitEvent(s_out, ev(STEPPED, k), 0));
                f(cudaMemcpyAsync(dst + a, qn + a, bytes, cudaMemcpyDefault, s_out));
            }
            f(cudaEventRecord(ev(LEFT, k), s_out));
        }
        std::swap(src, dst);
        std::swap(q, qn);
    }
    for (cudaStream_t s : h.streams) {   // also after a failure: what was enqueued is joined
        f(cudaEventRecord(h.events[0], s));
        f(cudaStreamWaitEvent(comp, h.events[0], 0));
    }
    return f.rc != CLAW_OK ? f.rc : cuda_rc(f.e);
}
