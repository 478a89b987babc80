// api.cu -- C ABI of the decoder: stream parsing and upload, decode
// orchestration, inspection hooks and per-kernel event timing.
//
// Stream layout (little endian):
//   header (128 bytes)  magic "WVS1", version 1, luma width/height, planes,
//                       chroma_420, levels, wavelet, num_frames, tlevels,
//                       block, quantiser, step, blocks per frame, number of
//                       stored blocks, byte offsets of table and payload.
//                       (Sec. 3.4: the header gives the number of frames, the
//                       frame size and the number of wavelet levels.)
//   block table         int32 [num_frames][blocks per frame]: slot of the
//                       block's coefficients in the payload, -1 when the block
//                       is all zero (the per-block BlockEnd pointers of Sec.
//                       3.4, here one fixed-size slot per stored block).
//   payload             int16 [slots][block][block], row-major blocks.
// Blocks of one coefficient frame: plane by plane; in each plane LL_L, then
// for l = L..1 the subbands HL_l, LH_l, HH_l (level-wise from the lowest
// frequency, Sec. 3.4), each cut into block x block tiles in row-major order.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "wv_impl.h"

using namespace wv;

namespace {

enum Kernel { kKFootprint = 0, kKTiles = 1, kKCoarse = 2, kKFine = 3, kKResample = 4 };

// Geometry of the stream's viewport and whole-plane decodes in its current
// decode mode: 0 = the default geometry (strip tiles for the streams the
// strip kernel decodes), 1 and 2 = square tiles.
const Geom &active_geom(const wv_stream *s) { return s->decode_mode == 0 ? s->g : s->gsq; }
// Strip fine pass (levels 2 and 1 streamed down strips, strip.cu).
bool strip_mode(const wv_stream *s) { return s->decode_mode == 0 && s->g.strip; }
// Coarse pass (levels L..3 into LL_2 planes) before the fine pass.
bool split_mode(const wv_stream *s) { return s->decode_mode != 1 && s->g.levels >= 3; }

// Coefficient frames of `frame` with the byte quantiser's parameters of the
// paper-faithful format (quant 1).
Bands stream_bands(const wv_stream *s, int frame) {
    Bands b = frame_bands(s->g, frame);
    if (s->g.quant == 1)
        for (int k = 0; k < b.n; ++k)
            for (int p = 0; p < 3; ++p)
                for (int c = 0; c < 2; ++c)
                    for (int e = 0; e < 2; ++e)
                        b.qp[k][p][c][e] = s->qp_host[(((size_t)b.t[k] * 3 + p) * 2 + c) * 2 + e];
    return b;
}

// Generation stamp of the next viewport (0 is never used: the stamp arrays
// start zeroed).
uint32_t next_gen(wv_stream *s) {
    s->gen = s->gen + 1 == 0 ? 1 : s->gen + 1;
    return s->gen;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

int parse(const void *bytes, size_t n, wv_stream_desc *d, StreamHeader *h) {
    if (!bytes || n < kHeaderBytes) return WV_ERR_FORMAT;
    memcpy(h, bytes, sizeof(StreamHeader));
    if (memcmp(h->magic, "WVS1", 4) != 0 || h->version != 1) return WV_ERR_FORMAT;
    d->width = (int)h->width;
    d->height = (int)h->height;
    d->planes = (int)h->planes;
    d->chroma_420 = (int)h->c420;
    d->levels = (int)h->levels;
    d->wavelet = (int)h->wavelet;
    d->num_frames = (int)h->num_frames;
    d->tlevels = (int)h->tlevels;
    d->block = (int)h->block;
    d->quant = (int)h->quant;
    d->step = h->step;
    d->stereo = (int)h->reserved0;
    Geom g;
    if (build_geom(*d, &g) != WV_OK) return WV_ERR_FORMAT;
    if ((int)h->nbpf != g.nbpf) return WV_ERR_FORMAT;
    const uint64_t tbytes = (uint64_t)g.num_frames * g.nbpf * 4;
    const uint64_t bsz = (uint64_t)g.block * g.block * 2;
    if (h->table_off < kHeaderBytes || h->table_off + tbytes > n) return WV_ERR_FORMAT;
    if (h->payload_off % 2 || h->payload_off < h->table_off + tbytes) return WV_ERR_FORMAT;
    if (h->n_payload > (n - std::min<uint64_t>(n, h->payload_off)) / bsz) return WV_ERR_FORMAT;
    const int32_t *tab = reinterpret_cast<const int32_t *>((const char *)bytes + h->table_off);
    for (uint64_t i = 0; i < (uint64_t)g.num_frames * g.nbpf; ++i) {
        int32_t s;
        memcpy(&s, tab + i, 4);
        if (s < -1 || (int64_t)s >= (int64_t)h->n_payload) return WV_ERR_FORMAT;
    }
    return WV_OK;
}

// Both geometries of a stream: square tiles always, strip tiles where the
// strip kernel applies (else a copy of the square geometry).
int stream_geoms(const wv_stream_desc &d, uint64_t n_payload, Geom *g, Geom *gsq) {
    const int rc = build_geom(d, gsq);
    if (rc != WV_OK) return rc;
    gsq->n_blocks = (int)std::min<uint64_t>(n_payload, 0x7fffffff);
    if (strip_eligible(d, n_payload)) {
        const int strips = viewable_strips(d);
        const int rs = strips <= kFineStrips ? build_geom_strip(d, g, 32, 32) : build_geom_strip(d, g);
        g->halves = strips <= kFineStrips / 4;
        g->n_blocks = gsq->n_blocks;
        return rs;
    }
    *g = *gsq;
    return WV_OK;
}

struct Layout {
    size_t payload, table, mask, err, total;
    int n_sets;
    struct Set {
        size_t recon[3], ll2[3], tiles, ctiles, tile_gen, ctile_gen, counters, end;
    } set[kViewSets];   // the buffers of the viewports in flight
};

// Device layout of a stream with at most max_sets buffer sets; tile lists and
// stamps hold the larger tile count of the two geometries.
Layout layout(const Geom &g0, const Geom &gsq, uint64_t n_payload, int max_sets) {
    Geom g = g0;
    g.total_tiles = std::max(g0.total_tiles, gsq.total_tiles);
    // tile lists: an edge strip is listed as two half strips
    const size_t list_tiles = std::max<size_t>(2 * (size_t)g0.total_tiles, gsq.total_tiles);
    Layout L;
    size_t o = 0;
    L.payload = o;
    o = align256(o + n_payload * g.block * g.block * 2);
    L.table = o;
    o = align256(o + (size_t)g.num_frames * g.nbpf * 4);
    L.mask = o;
    o = align256(o + (size_t)g.cells_x * g.cells_y);
    L.err = o;
    o = align256(o + 64);
    // one viewport at a time without a coarse pass (decode_region)
    L.n_sets = std::min(max_sets, g.levels < 3 ? 1 : g.strip && g.th == 32 ? kViewSets : kViewSetsLarge);
    for (int k = 0; k < L.n_sets; ++k) {
        Layout::Set &S = L.set[k];
        for (int p = 0; p < 3; ++p) {
            S.recon[p] = o;
            if (p < g.planes) o = align256(o + (size_t)g.p[p].w * g.p[p].h);
        }
        for (int p = 0; p < 3; ++p) {
            S.ll2[p] = o;
            if (p < g.planes && g.levels >= 3)
                o = align256(o + (size_t)g.p[p].ll2_pitch * (g.p[p].h >> 2) * 4);
        }
        S.tiles = o;
        o = align256(o + list_tiles * 4);
        S.ctiles = o;
        o = align256(o + (size_t)(g.total_ctiles > 0 ? g.total_ctiles : 1) * 4);
        S.tile_gen = o;
        o = align256(o + (size_t)g.total_tiles * 4);
        S.ctile_gen = o;
        o = align256(o + (size_t)(g.total_ctiles > 0 ? g.total_ctiles : 1) * 4);
        S.counters = o;
        o = align256(o + 64);
        S.end = o;
    }
    L.total = o;
    return L;
}

int cuda_err(cudaError_t e) { return e == cudaSuccess ? WV_OK : WV_ERR_CUDA; }

std::atomic<int> g_fail_allocs{0};   // device allocations still to fail (test hook)

void prof_begin(wv_stream *s, int kind) {
    if (!s->prof) return;
    if (s->ev_used + 2 > s->ev_pool.size()) {
        for (int i = 0; i < 64; ++i) {
            cudaEvent_t e;
            cudaEventCreate(&e);
            s->ev_pool.push_back(e);
        }
    }
    cudaEventRecord(s->ev_pool[s->ev_used], s->cs);
    s->ev_kind.push_back(kind);
}

void prof_end(wv_stream *s) {
    if (!s->prof) return;
    cudaEventRecord(s->ev_pool[s->ev_used + 1], s->cs);
    s->ev_used += 2;
}

int check_image(const wv_image *o) {
    if (!o || !o->dptr || o->width <= 0 || o->height <= 0 ||
        o->pitch_bytes < (size_t)o->width * 4 || (o->pitch_bytes % 4) != 0 ||
        ((uintptr_t)o->dptr % 4) != 0)
        return WV_ERR_ARG;
    return WV_OK;
}

// Tile decode of the selected tiles: a coarse pass (levels L..3 into LL_2
// planes) followed by a fine pass (levels 2 and 1), or all levels in one
// pass when the stream has fewer than three levels or mode 1 is set.
// The fine pass (levels 2 and 1) of the listed tiles: strips, or square tiles
// reading LL_2 from the planes.
cudaError_t launch_fine(wv_stream *s, const Bands &b, const float *const *ll2, uint8_t *const *out_u8,
                        float *f32, int f32_plane, const uint32_t *tiles, int *counters,
                        cudaStream_t cs, int all_plane = -1) {
    const Geom &g = active_geom(s);
    if (strip_mode(s)) {
        // into the stream's reconstruction planes: chroma in alternating Cb, Cr groups
        bool own = false;
        for (int k = 0; k < s->n_sets; ++k)
            own = own || (out_u8[1] == s->set[k].recon[1] && out_u8[2] == s->set[k].recon[2]);
        const bool pairs = own && recon_pairs(s);
        uint8_t *const outs[3] = {out_u8[0], out_u8[1], pairs ? out_u8[1] + 4 : out_u8[2]};
        return launch_decode_strips(g, s->payload, s->table, b, ll2, s->ll2_pitch, outs, f32, f32_plane, tiles,
                                    counters, s->err, cs, pairs, all_plane);
    }
    return launch_decode_fine(g, s->payload, s->table, b, ll2, s->ll2_pitch, out_u8, f32, f32_plane, tiles,
                              counters, s->err, cs);
}

cudaError_t run_decode(wv_stream *s, const Bands &b, uint8_t *const *out_u8, float *f32,
                       int f32_plane, int all_plane = -1) {
    const Geom &g = active_geom(s);
    const ViewSet &S = s->set[0];
    cudaError_t e;
    if (split_mode(s)) {
        prof_begin(s, kKCoarse);
        e = launch_decode_coarse(g, s->payload, s->table, b, S.ll2, s->ll2_pitch, S.ctiles,
                                 S.counters + 1, s->err, s->cs, all_plane);
        prof_end(s);
        if (e != cudaSuccess) return e;
        const float *ll2c[3] = {S.ll2[0], S.ll2[1], S.ll2[2]};
        prof_begin(s, kKFine);
        e = launch_fine(s, b, ll2c, out_u8, f32, f32_plane, S.tiles, S.counters, s->cs, all_plane);
        prof_end(s);
        return e;
    }
    prof_begin(s, kKFine);
    e = launch_decode_tiles(g, s->payload, s->table, b, out_u8, f32, f32_plane, S.tiles, S.counters, s->err,
                            s->cs);
    prof_end(s);
    return e;
}

}  // namespace

namespace wv {

// Steps 1-3 of a viewport decode: footprint, tile lists and the tile decode
// of the region an out_w x out_h viewport reads (into the stream's
// reconstruction planes).
int eye_view(const Geom &g, int eye, int *row0, int *rows) {
    if (eye < 0 || eye > (g.stereo ? 1 : 0)) return WV_ERR_ARG;
    *rows = g.stereo ? g.p[0].h / 2 : g.p[0].h;
    *row0 = eye * *rows;
    return WV_OK;
}

// Internal streams and their events, handed from closed streams to new ones
// (making them took 60 us of a new stream's first decode).  At most kLanesKept
// idle ones per device while a wv_stream is open there, none once the last one
// is closed; nothing in flight uses an idle one.
struct Lane {
    cudaStream_t st = nullptr;
    cudaEvent_t fine = nullptr, free = nullptr;
};
constexpr size_t kLanesKept = 16;
struct DeviceLanes {
    int open = 0;   // open wv_streams of the device
    std::vector<Lane> idle;
};
std::mutex g_lane_mutex;
std::map<int, DeviceLanes> &device_lanes() {
    static auto *m = new std::map<int, DeviceLanes>();   // outlives every stream
    return *m;
}

void destroy_lane(const Lane &l) {
    if (l.st) cudaStreamDestroy(l.st);
    for (cudaEvent_t e : {l.fine, l.free})
        if (e) cudaEventDestroy(e);
}

// A stream of the device was opened, or closed (its lanes already given back).
void count_open(int device) {
    std::lock_guard<std::mutex> lock(g_lane_mutex);
    DeviceLanes &D = device_lanes()[device];
    D.idle.reserve(kLanesKept);   // give_lane never allocates
    D.open += 1;
}
void count_closed(int device) {
    std::vector<Lane> last;
    {
        std::lock_guard<std::mutex> lock(g_lane_mutex);
        DeviceLanes &D = device_lanes()[device];
        if (--D.open == 0) last.swap(D.idle);
    }
    for (const Lane &l : last) destroy_lane(l);
}

cudaError_t take_lane(int device, Lane *l) {
    {
        std::lock_guard<std::mutex> lock(g_lane_mutex);
        std::vector<Lane> &v = device_lanes()[device].idle;
        if (!v.empty()) {
            *l = v.back();
            v.pop_back();
            return cudaSuccess;
        }
    }
    *l = Lane{};
    cudaError_t e = cudaEventCreateWithFlags(&l->fine, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&l->free, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&l->st, cudaStreamNonBlocking);
    if (e != cudaSuccess) destroy_lane(*l);
    return e;
}

void give_lane(int device, const Lane &l) {
    {
        std::lock_guard<std::mutex> lock(g_lane_mutex);
        std::vector<Lane> &v = device_lanes()[device].idle;
        if (v.size() < kLanesKept) {
            v.push_back(l);
            return;
        }
    }
    destroy_lane(l);
}

int idle_lanes(int device) {
    std::lock_guard<std::mutex> lock(g_lane_mutex);
    const auto it = device_lanes().find(device);
    return it == device_lanes().end() ? 0 : (int)it->second.idle.size();
}

// The internal stream and events of set k (when it is first used).  The set's
// first chain waits for everything enqueued on cs so far: work on cs uses set
// 0.
cudaError_t ensure_set(wv_stream *s, int k) {
    ViewSet &S = s->set[k];
    if (S.st) return cudaSuccess;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && dev != s->device) return cudaErrorInvalidDevice;   // a new lane would be the other device's
    Lane l;
    if (e == cudaSuccess) e = take_lane(s->device, &l);
    if (e == cudaSuccess && (e = cudaEventRecord(l.free, s->cs)) != cudaSuccess) give_lane(s->device, l);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    S.st = l.st;
    S.fine = l.fine;
    S.free = l.free;
    return cudaSuccess;
}

void release_set(wv_stream *s, int k) {
    ViewSet &S = s->set[k];
    if (!S.st) return;
    cudaStreamSynchronize(S.st);
    give_lane(s->device, Lane{S.st, S.fine, S.free});
    S.st = nullptr;
    S.fine = S.free = nullptr;
}

// A stream that is ever captured into a CUDA graph decodes serially from
// then on: the internal stream is not part of a capture, and graph replays
// must not race with overlapped calls.
void check_capture(wv_stream *s) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s->cs, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        s->overlap = false;
    }
}

// After work on cs that used the per-viewport buffers of set 0: later
// overlapped viewports wait for it before reusing any set.
void mark_sets_used(wv_stream *s) {
    check_capture(s);
    if (!s->overlap) return;
    for (int k = 0; k < s->n_sets; ++k)
        if (s->set[k].st) cudaEventRecord(s->set[k].free, s->cs);
}

// Overlapped viewport decode into buffer set k: the whole chain on the set's
// stream, once the resampling of the set's previous viewport has read its
// reconstruction; cs waits for the chain, and the caller's resampling then
// runs on cs beside the next viewports' chains.
int decode_region_overlapped(wv_stream *s, const View &v, const Bands &b, uint32_t gen) {
    const Geom &g = active_geom(s);
    const int k = s->slot;
    s->slot = (k + 1) % s->n_sets;
    ViewSet &S = s->set[k];
    cudaError_t e = cudaStreamWaitEvent(S.st, S.free, 0);
    if (e != cudaSuccess) return WV_ERR_CUDA;
    launch_footprint(g, v, nullptr, S.tile_gen, S.ctile_gen, gen, S.counters, S.st);
    launch_select_tiles(g, S.tile_gen, S.ctile_gen, gen, S.tiles, S.ctiles, S.counters, S.st);
    e = launch_decode_coarse(g, s->payload, s->table, b, S.ll2, s->ll2_pitch, S.ctiles, S.counters + 1, s->err, S.st);
    const float *ll2c[3] = {S.ll2[0], S.ll2[1], S.ll2[2]};
    if (e == cudaSuccess) e = launch_fine(s, b, ll2c, S.recon, nullptr, -1, S.tiles, S.counters, S.st);
    if (e == cudaSuccess) e = cudaEventRecord(S.fine, S.st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s->cs, S.fine, 0);
    s->cur = k;
    s->pending = true;
    return e == cudaSuccess ? WV_OK : WV_ERR_CUDA;
}

// A whole plane into the caller's buffer: the coarse pass, which reads nothing
// but the stream, on the set's stream, so that it runs beside what is still on
// cs (the fine pass of the previous plane); the fine pass on cs, in order with
// the caller's other uses of the buffer.  Three planes of a 4096^2 frame as
// floats: 213 -> 182 us, a 512^2 grey frame 35 -> 27.
int decode_full_overlapped(wv_stream *s, const Bands &b, uint8_t *const *outs, float *f32, int plane) {
    const Geom &g = active_geom(s);
    ViewSet &S = s->set[s->slot];
    s->slot = (s->slot + 1) % s->n_sets;
    cudaError_t e = cudaStreamWaitEvent(S.st, S.free, 0);
    if (e == cudaSuccess)
        e = launch_decode_coarse(g, s->payload, s->table, b, S.ll2, s->ll2_pitch, S.ctiles, S.counters + 1, s->err,
                                 S.st, plane);
    if (e == cudaSuccess) e = cudaEventRecord(S.fine, S.st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s->cs, S.fine, 0);
    const float *ll2c[3] = {S.ll2[0], S.ll2[1], S.ll2[2]};
    if (e == cudaSuccess)
        e = launch_fine(s, b, ll2c, outs, f32, f32 ? plane : -1, S.tiles, S.counters, s->cs, plane);
    const cudaError_t e1 = cudaEventRecord(S.free, s->cs);
    return e == cudaSuccess && e1 == cudaSuccess ? WV_OK : WV_ERR_CUDA;
}

int decode_region(wv_stream *s, int frame, float yaw, float pitch, float fov, int out_w, int out_h, int eye) {
    const Geom &g = active_geom(s);
    int row0, rows;
    if (eye_view(g, eye, &row0, &rows) != WV_OK) return WV_ERR_ARG;
    const View v = make_view(yaw, pitch, fov, out_w, out_h, g.p[0].w, rows, row0);
    const Bands b = stream_bands(s, frame);
    const uint32_t gen = next_gen(s);
    check_capture(s);
    if (split_mode(s) && !s->prof && s->overlap && ensure_set(s, s->slot) == cudaSuccess)
        return decode_region_overlapped(s, v, b, gen);
    prof_begin(s, kKFootprint);
    ViewSet &S = s->set[0];
    launch_footprint(g, v, s->mask, S.tile_gen, S.ctile_gen, gen, S.counters, s->cs);
    prof_end(s);
    prof_begin(s, kKTiles);
    launch_select_tiles(g, S.tile_gen, S.ctile_gen, gen, S.tiles, S.ctiles, S.counters, s->cs);
    prof_end(s);
    const cudaError_t e = run_decode(s, b, S.recon, nullptr, -1);
    mark_sets_used(s);
    s->cur = 0;
    s->pending = true;
    return e == cudaSuccess ? WV_OK : WV_ERR_CUDA;
}

uint8_t *const *recon_planes(const wv_stream *s) { return s->set[s->cur].recon; }

void release_recon(wv_stream *s, bool again) {
    if (!s->pending && !again) return;
    s->pending = false;
    if (s->set[s->cur].st && s->overlap) cudaEventRecord(s->set[s->cur].free, s->cs);
}

}  // namespace wv

namespace {

int decode_viewport(wv_stream *s, int frame, float yaw, float pitch, float fov,
                    const wv_image *out, int eye = 0) {
    if (!s) return WV_ERR_ARG;
    if (frame < 0 || frame >= s->g.num_frames) return WV_ERR_ARG;
    if (!(fov > 0.f && fov < 3.14159f) || !isfinite(yaw) || !isfinite(pitch)) return WV_ERR_ARG;
    if (check_image(out) != WV_OK) return WV_ERR_ARG;
    const Geom &g = s->g;
    int row0, rows;
    if (eye_view(g, eye, &row0, &rows) != WV_OK) return WV_ERR_ARG;
    const int rc = wv::decode_region(s, frame, yaw, pitch, fov, out->width, out->height, eye);
    if (rc != WV_OK) return rc;
    const View v = make_view(yaw, pitch, fov, out->width, out->height, g.p[0].w, rows, row0);
    prof_begin(s, kKResample);
    launch_resample(g, v, recon_planes(s), nullptr, (uint8_t *)out->dptr, out->pitch_bytes, s->cs, nullptr,
                    nullptr, nullptr, recon_pairs(s), s->err);
    prof_end(s);
    release_recon(s);
    return cuda_err(cudaGetLastError());
}

// ---- host-side dependency cone (accounting only) ----

void dilate_axis(const std::vector<uint8_t> &in, std::vector<uint8_t> &out, int w, int h,
                 bool along_x, int wavelet) {
    out.assign(in.size(), 0);
    const int n = along_x ? w : h;
    auto refl = [n](int i) {
        if (n == 1) return 0;
        const int period = 2 * (n - 1);
        i %= period;
        if (i < 0) i += period;
        return i >= n ? period - i : i;
    };
    // synthesis output i reads interleaved inputs i-3..i+3 (even i) or i-4..i+4
    // (odd i) for 9/7, i-1..i+1 or i-2..i+2 for 5/3
    const int se = wavelet == WV_WAVELET_97 ? 3 : 1;
    const int so = wavelet == WV_WAVELET_97 ? 4 : 2;
    for (int y = 0; y < h; ++y) {
        for (int x = 0; x < w; ++x) {
            if (!in[(size_t)y * w + x]) continue;
            const int i = along_x ? x : y;
            const int r = (i & 1) ? so : se;
            for (int o = -r; o <= r; ++o) {
                const int j = refl(i + o);
                if (along_x) out[(size_t)y * w + j] = 1;
                else out[(size_t)j * w + x] = 1;
            }
        }
    }
}

// fbits: optional foveation bits per mask cell (bit l - 1 keeps the details
// of level l = 1, 2); dropped coefficients are not read.
unsigned long long cone_bytes(const wv_stream *s, int frame, const uint8_t *mask,
                              const uint8_t *fbits = nullptr, unsigned long long *fine_part = nullptr) {
    const Geom &g = s->g;
    const Bands b = frame_bands(g, frame);
    unsigned long long total = 0, fine = 0;
    for (int p = 0; p < g.planes; ++p) {
        const PlaneGeom &pg = g.p[p];
        int w = pg.w, h = pg.h;
        const int cell = kCell / pg.sub;
        std::vector<uint8_t> R((size_t)w * h), X, tmp;
        for (int y = 0; y < h; ++y)
            for (int x = 0; x < w; ++x)
                R[(size_t)y * w + x] = mask[(size_t)(y / cell) * g.cells_x + x / cell] ? 1 : 0;
        auto count = [&](int level, int sub, int kx, int ky) {
            if (fbits && level <= 2 && sub != 0) {
                const int X = (kx << level) * pg.sub, Y = (ky << level) * pg.sub;
                if (!((fbits[(size_t)(Y / kCell) * g.cells_x + X / kCell] >> (level - 1)) & 1)) return;
            }
            const int bid = pg.base[level][sub] + (ky >> g.log2b) * pg.nbx[level] + (kx >> g.log2b);
            for (int k = 0; k < b.n; ++k)
                if (s->table_host[(size_t)b.t[k] * g.nbpf + bid] >= 0) {
                    total += 2;
                    if (level <= 2 && (sub != 0 || level < g.levels || g.levels <= 2)) fine += 2;
                }
        };
        for (int l = 1; l <= g.levels; ++l) {
            dilate_axis(R, tmp, w, h, true, g.wavelet);
            dilate_axis(tmp, X, w, h, false, g.wavelet);
            std::vector<uint8_t> next((size_t)(w / 2) * (h / 2));
            for (int y = 0; y < h; ++y)
                for (int x = 0; x < w; ++x) {
                    if (!X[(size_t)y * w + x]) continue;
                    const int sub = (x & 1) + 2 * (y & 1);
                    if (sub == 0) next[(size_t)(y >> 1) * (w / 2) + (x >> 1)] = 1;
                    else count(l, sub, x >> 1, y >> 1);
                }
            R.swap(next);
            w /= 2;
            h /= 2;
        }
        for (int y = 0; y < h; ++y)
            for (int x = 0; x < w; ++x)
                if (R[(size_t)y * w + x]) count(g.levels, 0, x, y);
    }
    if (fine_part) *fine_part = fine;
    return total;
}

// Foveation bits of every mask cell in double precision (the same definition
// as the device footprint: cell centre direction, viewer angles, max norm).
void fovea_bits_host(const Geom &g, double yaw, double pitch, const wv_request &r,
                     std::vector<uint8_t> &out) {
    const double pi = 3.14159265358979323846;
    const double cy = cos(yaw), sy = sin(yaw), cp = cos(pitch), sp = sin(pitch);
    const double R[9] = {cy, -sy * sp, sy * cp, 0.0, cp, sp, -sy, -cy * sp, cy * cp};
    out.assign((size_t)g.cells_x * g.cells_y, 0);
    for (int j = 0; j < g.cells_y; ++j)
        for (int i = 0; i < g.cells_x; ++i) {
            const double lon = 2.0 * pi * ((i + 0.5) * kCell / g.p[0].w - 0.5);
            const double lat = pi * (0.5 - (j + 0.5) * kCell / g.p[0].h);
            const double d[3] = {cos(lat) * sin(lon), sin(lat), cos(lat) * cos(lon)};
            const double x = R[0] * d[0] + R[3] * d[1] + R[6] * d[2];
            const double y = R[1] * d[0] + R[4] * d[1] + R[7] * d[2];
            const double z = R[2] * d[0] + R[5] * d[1] + R[8] * d[2];
            if (!(z > 0.0)) continue;
            const double dist = std::max(fabs(atan2(x, z) - r.gaze_x), fabs(atan2(y, z) - r.gaze_y));
            out[(size_t)j * g.cells_x + i] = (uint8_t)((dist <= r.r1 ? 1 : 0) | (dist <= r.r2 ? 2 : 0));
        }
}

}  // namespace

// ---------------------------------------------------------------------------
// geometry helpers
// ---------------------------------------------------------------------------

namespace wv {

cudaError_t dev_alloc(void **p, size_t bytes) {
    int n = g_fail_allocs.load();
    while (n > 0) {
        if (g_fail_allocs.compare_exchange_weak(n, n - 1)) return cudaErrorMemoryAllocation;
    }
    return cudaMalloc(p, bytes);
}

cudaError_t opt_in_smem(const void *fn, int bytes) {
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, int> opted;   // (kernel, device) -> bytes set
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    int &have = opted[std::make_pair(fn, dev)];
    if (bytes <= have) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) have = bytes;
    return e;
}

bool recon_pairs(const wv_stream *s) { return s->pair_ok && s->decode_mode == 0 && s->g.strip; }

namespace {

// Common geometry of both tile organisations: output tiles tw x th (plane
// pixels, multiples of the 32-pixel mask cell, and of 16 chroma pixels) and
// coarse tiles of ctile LL_2 samples.
int build_geom_tiles(const wv_stream_desc &d, Geom *g, int tw, int th, int strip, int ctile) {
    memset(g, 0, sizeof(*g));
    if (tw % kCell || th % kCell || tw <= 0 || th <= 0 || (ctile != 32 && ctile != 64)) return WV_ERR_ARG;
    if (d.planes != 1 && d.planes != 3) return WV_ERR_ARG;
    if (d.chroma_420 != 0 && d.chroma_420 != 1) return WV_ERR_ARG;
    if (d.levels < 1 || d.levels > kMaxLevels) return WV_ERR_ARG;
    if (d.wavelet != WV_WAVELET_53 && d.wavelet != WV_WAVELET_97) return WV_ERR_ARG;
    if (d.tlevels < 0 || d.tlevels > kMaxBands - 1) return WV_ERR_ARG;
    if (d.num_frames < 1 || d.num_frames % (1 << d.tlevels)) return WV_ERR_ARG;
    if (d.block < 16 || d.block > 256 || (d.block & (d.block - 1))) return WV_ERR_ARG;
    if (d.quant != 0 && d.quant != 1) return WV_ERR_ARG;
    if (d.quant == 1 && (d.wavelet != WV_WAVELET_97 || d.block != 32)) return WV_ERR_ARG;
    if (!(d.step > 0.f) || !isfinite(d.step)) return WV_ERR_ARG;
    if (d.wavelet == WV_WAVELET_53 && (d.step != floorf(d.step) || d.step > 65536.f))
        return WV_ERR_ARG;
    if (d.width < 2 || d.height < 2 || d.width > 16384 || d.height > 16384) return WV_ERR_ARG;
    if (d.stereo != 0 && d.stereo != 1) return WV_ERR_ARG;
    if (d.stereo && d.height % (2 * kCell)) return WV_ERR_ARG;
    if (d.width % kCell || d.height % kCell) return WV_ERR_ARG;
    g->planes = d.planes;
    g->c420 = d.planes == 3 ? d.chroma_420 : 0;
    g->levels = d.levels;
    g->wavelet = d.wavelet;
    g->num_frames = d.num_frames;
    g->tlevels = d.tlevels;
    g->block = d.block;
    g->log2b = 0;
    while ((1 << g->log2b) < d.block) ++g->log2b;
    g->step = d.step;
    g->quant = d.quant;
    g->stereo = d.stereo;
    g->cells_x = d.width / kCell;
    g->cells_y = d.height / kCell;
    g->tw = tw;
    g->th = th;
    g->strip = strip;
    g->ctile = ctile;
    // LL_2 window of an output tile: the square tile kernel's fine pass reads
    // its LL_2 window q t - 3 .. q t + q + 2 (q = tile / 4, the 9/7 halo of
    // two levels); a strip's level-2 lanes read LL_2 columns X0/4 - 4 ..
    // X0/4 + 59 and its level-2 row pairs LL_2 rows Y0/4 - 3 .. Y0/4 + th/4 + 2
    g->wx0 = strip ? -4 : -3;
    g->wx1 = strip ? 59 : tw / 4 + 2;
    g->wy0 = -3;
    g->wy1 = th / 4 + 2;
    int id = 0;
    g->total_tiles = 0;
    g->total_ctiles = 0;
    for (int p = 0; p < d.planes; ++p) {
        PlaneGeom &pg = g->p[p];
        pg.sub = (p > 0 && g->c420) ? 2 : 1;
        pg.w = d.width / pg.sub;
        pg.h = d.height / pg.sub;
        if (pg.w % (1 << d.levels) || pg.h % (1 << d.levels)) return WV_ERR_ARG;
        if ((pg.w >> d.levels) < 2 || (pg.h >> d.levels) < 2) return WV_ERR_ARG;
        for (int l = 1; l <= d.levels; ++l) {
            const int sw = pg.w >> l, sh = pg.h >> l;
            pg.nbx[l] = (sw + d.block - 1) / d.block;
            pg.nby[l] = (sh + d.block - 1) / d.block;
        }
        const int L = d.levels;
        pg.base[L][0] = id;
        id += pg.nbx[L] * pg.nby[L];
        for (int l = L; l >= 1; --l)
            for (int s = 1; s <= 3; ++s) {
                pg.base[l][s] = id;
                id += pg.nbx[l] * pg.nby[l];
            }
        pg.tiles_x = (pg.w + tw - 1) / tw;
        pg.tiles_y = (pg.h + th - 1) / th;
        g->total_tiles += pg.tiles_x * pg.tiles_y;
        pg.ll2_pitch = (((pg.w >> 2) + 7) / 8) * 8;
        if (d.levels >= 3) {
            pg.ctiles_x = ((pg.w >> 2) + ctile - 1) / ctile;
            pg.ctiles_y = ((pg.h >> 2) + ctile - 1) / ctile;
        }
        g->total_ctiles += pg.ctiles_x * pg.ctiles_y;
    }
    g->nbpf = id;
    return WV_OK;
}

}  // namespace

int build_geom(const wv_stream_desc &d, Geom *g, int tile, int ctile) {
    if (tile != 64 && tile != 128) {
        memset(g, 0, sizeof(*g));
        return WV_ERR_ARG;
    }
    return build_geom_tiles(d, g, tile, tile, 0, ctile);
}

int build_geom_rect(const wv_stream_desc &d, Geom *g, int tw, int th, int ctile) {
    if (tw < 64 || tw > 256 || th < 64 || th > 256) {
        memset(g, 0, sizeof(*g));
        return WV_ERR_ARG;
    }
    return build_geom_tiles(d, g, tw, th, 0, ctile);
}

// The strip kernel decodes levels 2 and 1 of streams of three or more levels
// (LL_2 from the coarse pass; taking it from the LL band of two-level streams
// in the same loop cost 5 % in spilled registers) and addresses the payload
// with 32-bit element offsets.
bool strip_eligible(const wv_stream_desc &d, uint64_t n_payload) {
    return d.levels >= 3 && (d.quant == 0 || d.wavelet == WV_WAVELET_97) &&
           n_payload * (uint64_t)d.block * (uint64_t)d.block < (1ull << 32);
}

int viewable_strips(const wv_stream_desc &d) {
    long long n = 0;
    for (int p = 0; p < d.planes; ++p) {
        const int sub = p > 0 && d.chroma_420 ? 2 : 1;
        n += ((d.width / sub + kStripW - 1) / kStripW) * (long long)((d.height / sub + 63) / 64);
    }
    return (int)std::min<long long>(n / (d.stereo ? 2 : 1), 0x7fffffff);
}

int build_geom_strip(const wv_stream_desc &d, Geom *g, int th, int ctile) {
    if (th % kCell || th < 32 || th > 256) {
        memset(g, 0, sizeof(*g));
        return WV_ERR_ARG;
    }
    return build_geom_tiles(d, g, kStripW, th, 1, ctile);
}

Bands frame_bands(const Geom &g, int frame) {
    Bands b;
    memset(&b, 0, sizeof(b));
    const int k = g.tlevels, n = 1 << k;
    const int set = frame / n, fl = frame % n;
    b.n = 1 + k;
    b.t[0] = set * n;
    b.bit[0] = 0;
    int idx = 1;
    for (int j = k; j >= 1; --j, ++idx) {
        b.t[idx] = set * n + (1 << (k - j)) + (fl >> j);
        b.bit[idx] = (fl >> (j - 1)) & 1;
    }
    for (; idx < kMaxBands; ++idx) {
        b.t[idx] = 0;
        b.bit[idx] = 0;
    }
    return b;
}

Frustum make_frustum(const View &v) {
    // camera-space normals of x <= T z, x >= -T z, y <= T z, y >= -T z
    const double T = v.t, nrm = 1.0 / sqrt(1.0 + T * T);
    const double m[4][3] = {{-nrm, 0.0, T * nrm}, {nrm, 0.0, T * nrm},
                            {0.0, -nrm, T * nrm}, {0.0, nrm, T * nrm}};
    Frustum f;
    for (int k = 0; k < 4; ++k)
        for (int i = 0; i < 3; ++i)
            f.n[k][i] = (float)(v.r[3 * i + 0] * m[k][0] + v.r[3 * i + 1] * m[k][1] +
                                v.r[3 * i + 2] * m[k][2]);
    return f;
}

View make_view(float yaw, float pitch, float fov, int out_w, int out_h, int eq_w, int eq_h, int row0) {
    const double cy = cos((double)yaw), sy = sin((double)yaw);
    const double cp = cos((double)pitch), sp = sin((double)pitch);
    // R = R_y(yaw) R_x(pitch); R_x: (x, y, z) -> (x, y cp + z sp, -y sp + z cp)
    const double R[9] = {cy, -sy * sp, sy * cp,
                         0.0, cp, sp,
                         -sy, -cy * sp, cy * cp};
    View v;
    for (int i = 0; i < 9; ++i) v.r[i] = (float)R[i];
    v.t = (float)tan((double)fov / 2.0);
    v.sx = (float)(2.0 / out_w);
    v.sy = (float)(2.0 / out_h);
    const double pi = 3.14159265358979323846;
    v.ku = (float)(eq_w / (2.0 * pi));
    v.cu = (float)(0.5 * eq_w - 0.5);
    v.kv = (float)(-eq_h / pi);
    v.cv = (float)(0.5 * eq_h - 0.5 + row0);
    v.out_w = out_w;
    v.out_h = out_h;
    v.row0 = row0;
    v.rows = eq_h;
    return v;
}

}  // namespace wv

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------

extern "C" {

const char *wv_strerror(int code) {
    switch (code) {
    case WV_OK: return "ok";
    case WV_ERR_ARG: return "invalid argument";
    case WV_ERR_FORMAT: return "malformed or unsupported stream";
    case WV_ERR_OOM: return "out of memory or buffer too small";
    case WV_ERR_CUDA: return "CUDA error or no CUDA device";
    case WV_ERR_RANGE: return "value out of range";
    case WV_ERR_TIMEOUT: return "device wait timed out";
    case WV_ERR_DEVICE: return "kernel reported an inconsistency";
    default: return "unknown error";
    }
}

int wv_stream_query(const void *bytes, size_t n, wv_stream_desc *desc, size_t *device_bytes) {
    return wv_stream_query_ex(bytes, n, 0, desc, device_bytes);
}

int wv_stream_query_ex(const void *bytes, size_t n, int flags, wv_stream_desc *desc, size_t *device_bytes) {
    return query_stream(bytes, n, flags, kViewSets, desc, device_bytes);
}

int wv_open_stream(const void *bytes, size_t n, void *device_mem, size_t device_bytes,
                   void *cuda_stream, wv_stream **out) {
    return wv_open_stream_ex(bytes, n, device_mem, device_bytes, cuda_stream, 0, out);
}

int wv_open_stream_ex(const void *bytes, size_t n, void *device_mem, size_t device_bytes,
                      void *cuda_stream, int flags, wv_stream **out) {
    return open_stream(bytes, n, device_mem, device_bytes, cuda_stream, flags, kViewSets, out);
}

}  // extern "C"

namespace wv {

int query_stream(const void *bytes, size_t n, int flags, int max_sets, wv_stream_desc *desc, size_t *device_bytes) {
    if (flags & ~WV_OPEN_HOST_PAYLOAD) return WV_ERR_ARG;
    const bool host_payload = (flags & WV_OPEN_HOST_PAYLOAD) != 0;
    wv_stream_desc d;
    StreamHeader h;
    if (is_paper_stream(bytes, n)) {
        PaperInfo info;
        const int rc = paper_parse(bytes, n, &d, &info);
        if (rc != WV_OK) return rc;
        if (desc) *desc = d;
        if (device_bytes) {
            Geom g, gsq;
            stream_geoms(d, info.n_slots, &g, &gsq);
            *device_bytes = layout(g, gsq, host_payload ? 0 : info.n_slots, max_sets).total;
        }
        return WV_OK;
    }
    const int rc = parse(bytes, n, &d, &h);
    if (rc != WV_OK) return rc;
    if (desc) *desc = d;
    if (device_bytes) {
        Geom g, gsq;
        stream_geoms(d, h.n_payload, &g, &gsq);
        *device_bytes = layout(g, gsq, host_payload ? 0 : h.n_payload, max_sets).total;
    }
    return WV_OK;
}

int open_stream(const void *bytes, size_t n, void *device_mem, size_t device_bytes, void *cuda_stream, int flags,
                int max_sets, wv_stream **out) {
    if (!out) return WV_ERR_ARG;
    *out = nullptr;
    if (flags & ~WV_OPEN_HOST_PAYLOAD) return WV_ERR_ARG;
    const bool host_payload = (flags & WV_OPEN_HOST_PAYLOAD) != 0;
    wv_stream_desc d;
    StreamHeader h;
    PaperInfo paper;
    const bool is_paper = is_paper_stream(bytes, n);
    int rc = is_paper ? paper_parse(bytes, n, &d, &paper) : parse(bytes, n, &d, &h);
    if (rc != WV_OK) return rc;
    if (is_paper) {
        memset(&h, 0, sizeof(h));
        h.n_payload = paper.n_slots;
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return WV_ERR_CUDA;
    wv_stream *s = new (std::nothrow) wv_stream();
    if (!s) return WV_ERR_OOM;
    stream_geoms(d, h.n_payload, &s->g, &s->gsq);
    s->desc = d;
    cudaGetDevice(&s->device);
    s->cs = (cudaStream_t)cuda_stream;
    s->n_payload = h.n_payload;
    const Layout L = layout(s->g, s->gsq, host_payload ? 0 : h.n_payload, max_sets);
    const size_t payload_bytes = (size_t)h.n_payload * s->g.block * s->g.block * 2;
    if (host_payload && payload_bytes) {
        // the coefficient store in pinned, device-mapped host memory: the
        // tile decoder reads the blocks a viewport needs from there (on a
        // Grace-Blackwell node over NVLink-C2C) instead of an HBM copy
        if (cudaHostAlloc(&s->host_payload, payload_bytes, cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();
            delete s;
            return WV_ERR_OOM;
        }
        void *dp = nullptr;
        if (cudaHostGetDevicePointer(&dp, s->host_payload, 0) != cudaSuccess) {
            cudaGetLastError();
            cudaFreeHost(s->host_payload);
            delete s;
            return WV_ERR_CUDA;
        }
        s->payload = (int16_t *)dp;
    }
    if (device_mem) {
        if (device_bytes < L.total || ((uintptr_t)device_mem % 256)) {
            if (s->host_payload) cudaFreeHost(s->host_payload);
            delete s;
            return WV_ERR_OOM;
        }
        s->dmem = device_mem;
    } else {
        if (dev_alloc(&s->dmem, L.total) != cudaSuccess) {
            cudaGetLastError();
            if (s->host_payload) cudaFreeHost(s->host_payload);
            delete s;
            return WV_ERR_OOM;
        }
        s->owns = true;
    }
    s->dbytes = L.total;
    count_open(s->device);   // from here on the stream ends in wv_close_stream
    char *base = (char *)s->dmem;
    if (!host_payload) s->payload = (int16_t *)(base + L.payload);
    s->table = (int32_t *)(base + L.table);
    s->mask = (uint8_t *)(base + L.mask);
    s->err = (int *)(base + L.err);
    s->n_sets = L.n_sets;
    s->pair_ok = s->g.planes == 3;
    for (int k = 0; k < L.n_sets; ++k) {
        const Layout::Set &A = L.set[k];
        ViewSet &S = s->set[k];
        for (int p = 0; p < 3; ++p) {
            S.recon[p] = p < s->g.planes ? (uint8_t *)(base + A.recon[p]) : nullptr;
            S.ll2[p] = p < s->g.planes && s->g.levels >= 3 ? (float *)(base + A.ll2[p]) : nullptr;
        }
        S.tiles = (uint32_t *)(base + A.tiles);
        S.ctiles = (uint32_t *)(base + A.ctiles);
        S.tile_gen = (uint32_t *)(base + A.tile_gen);
        S.ctile_gen = (uint32_t *)(base + A.ctile_gen);
        S.counters = (int *)(base + A.counters);
        s->pair_ok = s->pair_ok && A.recon[2] == A.recon[1] + (size_t)s->g.p[1].w * s->g.p[1].h;
    }
    for (int p = 0; p < 3; ++p)
        s->ll2_pitch[p] = p < s->g.planes && s->g.levels >= 3 ? s->g.p[p].ll2_pitch : 0;
    const size_t tcount = (size_t)s->g.num_frames * s->g.nbpf;
    s->table_host.resize(tcount);
    if (is_paper) {
        memcpy(s->table_host.data(), paper.table.data(), tcount * 4);
        s->qp_host = paper.qp;
    } else {
        memcpy(s->table_host.data(), (const char *)bytes + h.table_off, tcount * 4);
    }
    cudaError_t e = cudaMemcpyAsync(s->table, s->table_host.data(), tcount * 4,
                                    cudaMemcpyHostToDevice, s->cs);
    if (e == cudaSuccess && is_paper)
        e = paper_transcode(bytes, n, paper, s->payload, s->cs);
    else if (e == cudaSuccess && h.n_payload && host_payload)
        memcpy(s->host_payload, (const char *)bytes + h.payload_off, payload_bytes);
    else if (e == cudaSuccess && h.n_payload)
        e = cudaMemcpyAsync(s->payload, (const char *)bytes + h.payload_off, payload_bytes,
                            cudaMemcpyHostToDevice, s->cs);
    // 9/7 dead-zone codes become t = 2q + sign(q) on the device when every
    // |q| <= kDzTMax (the tile decoder then needs no sign logic)
    if (e == cudaSuccess && !is_paper && h.n_payload && s->g.wavelet == WV_WAVELET_97 && s->g.quant == 0) {
        const size_t count = (size_t)h.n_payload * s->g.block * s->g.block;
        int max_abs = 0;
        e = cudaMemsetAsync(s->set[0].counters + 8, 0, 4, s->cs);
        if (e == cudaSuccess) e = payload_max_abs(s->payload, count, s->set[0].counters + 8, s->cs);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&max_abs, s->set[0].counters + 8, 4, cudaMemcpyDeviceToHost, s->cs);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->cs);
        if (e == cudaSuccess && max_abs <= kDzTMax) {
            e = payload_to_deadzone_t(s->payload, count, s->cs);
            s->g.dz_t = 1;
            s->gsq.dz_t = 1;
        }
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(base + L.mask, 0, L.total - L.mask, s->cs);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->cs);
    if (e != cudaSuccess) {
        cudaGetLastError();
        wv_close_stream(s);
        return WV_ERR_CUDA;
    }
    *out = s;
    return WV_OK;
}

}  // namespace wv

extern "C" {

void wv_debug_fail_device_allocs(int n) { g_fail_allocs.store(n > 0 ? n : 0); }

int wv_debug_idle_streams(int device) { return idle_lanes(device); }

int wv_set_cuda_stream(wv_stream *s, void *cuda_stream) {
    if (!s) return WV_ERR_ARG;
    s->cs = (cudaStream_t)cuda_stream;
    return WV_OK;
}

void wv_close_stream(wv_stream *s) {
    if (!s) return;
    cudaStreamSynchronize(s->cs);
    for (int k = 0; k < kViewSets; ++k) release_set(s, k);
    count_closed(s->device);
    if (s->host_payload) cudaFreeHost(s->host_payload);
    for (cudaEvent_t e : s->ev_pool) cudaEventDestroy(e);
    if (s->owns && s->dmem) cudaFree(s->dmem);
    delete s;
}

int wv_decode_viewport(wv_stream *s, int frame, float yaw, float pitch, float fov,
                       const wv_image *out) {
    return decode_viewport(s, frame, yaw, pitch, fov, out);
}

int wv_decode_viewport_eye(wv_stream *s, int frame, int eye, float yaw, float pitch, float fov,
                           const wv_image *out) {
    return decode_viewport(s, frame, yaw, pitch, fov, out, eye);
}

int wv_decode_full(wv_stream *s, int frame, int plane, void *dptr, int as_float) {
    if (!s || frame < 0 || frame >= s->g.num_frames || plane < 0 || plane >= s->g.planes)
        return WV_ERR_ARG;
    if (!dptr && as_float) return WV_ERR_ARG;
    if ((uintptr_t)dptr % (as_float ? 4 : 2)) return WV_ERR_ARG;   // the square tiles store byte pairs
    // Byte planes off a word boundary (strips store words) and float output of
    // streams the float strip kernels do not take run the square-tile passes
    // (the same arithmetic per sample).
    struct ModeGuard {
        wv_stream *s;
        int saved;
        ~ModeGuard() { s->decode_mode = saved; }
    } guard{s, s->decode_mode};
    if (strip_mode(s) && (as_float ? !strip_float_supported(s->g) : (uintptr_t)dptr % 4 != 0)) s->decode_mode = 2;
    const Geom &g = active_geom(s);
    const ViewSet &S = s->set[0];
    uint8_t *outs[3] = {S.recon[0], S.recon[1], S.recon[2]};
    float *f32 = nullptr;
    if (dptr) {
        if (as_float) f32 = (float *)dptr;
        else outs[plane] = (uint8_t *)dptr;
    }
    // strips: every tile of the plane, without lists (their count only serves
    // the profile)
    const int all_plane = strip_mode(s) ? plane : -1;
    check_capture(s);
    if (dptr && all_plane >= 0 && !s->prof && s->overlap && ensure_set(s, s->slot) == cudaSuccess)
        return decode_full_overlapped(s, stream_bands(s, frame), outs, f32, plane);
    if (all_plane < 0 || s->prof) launch_all_tiles(g, plane, S.tiles, S.counters, s->cs);
    if (all_plane < 0 && split_mode(s)) launch_all_ctiles(g, plane, S.ctiles, S.counters, s->cs);
    cudaError_t e = run_decode(s, stream_bands(s, frame), outs, f32, as_float ? plane : -1, all_plane);
    mark_sets_used(s);
    if (!dptr) {   // set 0's reconstruction now holds the decode (for wv_resample_at)
        s->cur = 0;
        s->pending = true;
    }
    if (e != cudaSuccess) return WV_ERR_CUDA;
    return cuda_err(cudaGetLastError());
}

int wv_stream_sync_status(wv_stream *s) {
    if (!s) return WV_ERR_ARG;
    if (cudaStreamSynchronize(s->cs) != cudaSuccess) return WV_ERR_CUDA;
    int err = 0;
    if (cudaMemcpy(&err, s->err, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return WV_ERR_CUDA;
    if (err) cudaMemset(s->err, 0, 4);
    return err;
}

int wv_debug_footprint(wv_stream *s, float yaw, float pitch, float fov, int out_w, int out_h,
                       uint8_t *mask_host, int *tiles) {
    if (!s || out_w <= 0 || out_h <= 0 || !(fov > 0.f && fov < 3.14159f)) return WV_ERR_ARG;
    const Geom &g = active_geom(s);
    int row0, rows;
    eye_view(g, 0, &row0, &rows);
    const View v = make_view(yaw, pitch, fov, out_w, out_h, g.p[0].w, rows, row0);
    uint8_t *m = s->mask;
    const uint32_t gen = next_gen(s);
    const ViewSet &S = s->set[0];
    launch_footprint(g, v, m, S.tile_gen, S.ctile_gen, gen, S.counters, s->cs);
    launch_select_tiles(g, S.tile_gen, S.ctile_gen, gen, S.tiles, S.ctiles, S.counters, s->cs);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && mask_host)
        e = cudaMemcpyAsync(mask_host, m, (size_t)g.cells_x * g.cells_y, cudaMemcpyDeviceToHost, s->cs);
    int cnt = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&cnt, S.counters, 4, cudaMemcpyDeviceToHost, s->cs);
    mark_sets_used(s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->cs);
    if (tiles) *tiles = cnt;
    return cuda_err(e);
}

int wv_debug_project(wv_stream *s, float yaw, float pitch, float fov, int out_w, int out_h,
                     float *uv_dev) {
    if (!s || !uv_dev || out_w <= 0 || out_h <= 0 || !(fov > 0.f && fov < 3.14159f))
        return WV_ERR_ARG;
    int row0, rows;
    eye_view(s->g, 0, &row0, &rows);
    const View v = make_view(yaw, pitch, fov, out_w, out_h, s->g.p[0].w, rows, row0);
    launch_project(v, uv_dev, s->cs);
    return cuda_err(cudaGetLastError());
}

int wv_resample_at(wv_stream *s, const float *uv_dev, const wv_image *out) {
    if (!s || !uv_dev || check_image(out) != WV_OK) return WV_ERR_ARG;
    View v = make_view(0.f, 0.f, 1.f, out->width, out->height, s->g.p[0].w, s->g.p[0].h);
    launch_resample(s->g, v, recon_planes(s), uv_dev, (uint8_t *)out->dptr, out->pitch_bytes, s->cs, nullptr,
                    nullptr, nullptr, recon_pairs(s), s->err);
    release_recon(s, true);   // any number of reads of the last decode: each releases its set again
    return cuda_err(cudaGetLastError());
}

int wv_cone_bytes(wv_stream *s, int frame, const uint8_t *mask_host, unsigned long long *bytes) {
    if (!s || !mask_host || !bytes || frame < 0 || frame >= s->g.num_frames) return WV_ERR_ARG;
    *bytes = cone_bytes(s, frame, mask_host);
    return WV_OK;
}

int wv_cone_bytes_split(wv_stream *s, int frame, const uint8_t *mask_host, unsigned long long *fine,
                        unsigned long long *coarse) {
    if (!s || !mask_host || !fine || !coarse || frame < 0 || frame >= s->g.num_frames) return WV_ERR_ARG;
    const unsigned long long total = cone_bytes(s, frame, mask_host, nullptr, fine);
    *coarse = total - *fine;
    return WV_OK;
}

int wv_cone_bytes_fovea(wv_stream *s, int frame, const uint8_t *mask_host,
                        const uint8_t *fovea_host, unsigned long long *bytes) {
    if (!s || !mask_host || !bytes || frame < 0 || frame >= s->g.num_frames) return WV_ERR_ARG;
    *bytes = cone_bytes(s, frame, mask_host, fovea_host);
    return WV_OK;
}

int wv_request_bytes(const wv_request *r, unsigned long long *cone, unsigned long long *region) {
    if (!r || !r->s || !cone || !region) return WV_ERR_ARG;
    wv_stream *s = r->s;
    const Geom &g = s->g;
    if (r->frame < 0 || r->frame >= g.num_frames || r->out.width <= 0 || r->out.height <= 0)
        return WV_ERR_ARG;
    std::vector<uint8_t> mask((size_t)g.cells_x * g.cells_y);
    int tiles = 0;
    const int rc = wv_debug_footprint(s, r->yaw, r->pitch, r->fov, r->out.width, r->out.height,
                                      mask.data(), &tiles);
    if (rc != WV_OK) return rc;
    std::vector<uint8_t> fb;
    if (r->fovea) fovea_bits_host(g, r->yaw, r->pitch, *r, fb);
    *cone = cone_bytes(s, r->frame, mask.data(), r->fovea ? fb.data() : nullptr);
    unsigned long long cells = 0;
    for (uint8_t m : mask) cells += m ? 1 : 0;
    unsigned long long per_cell = 0;
    for (int p = 0; p < g.planes; ++p) per_cell += (unsigned long long)(kCell / g.p[p].sub) * (kCell / g.p[p].sub);
    *region = cells * per_cell;
    return WV_OK;
}

int wv_profile_begin(wv_stream *s) {
    if (!s) return WV_ERR_ARG;
    s->prof = true;
    s->ev_used = 0;
    s->ev_kind.clear();
    return WV_OK;
}

int wv_profile_end(wv_stream *s, wv_profile *out) {
    if (!s || !out) return WV_ERR_ARG;
    memset(out, 0, sizeof(*out));
    if (cudaStreamSynchronize(s->cs) != cudaSuccess) return WV_ERR_CUDA;
    for (size_t i = 0; i < s->ev_kind.size(); ++i) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, s->ev_pool[2 * i], s->ev_pool[2 * i + 1]);
        const int k = s->ev_kind[i];
        out->ms[k] += ms;
        out->launches[k] += 1;
    }
    int cnt = 0;
    cudaMemcpy(&cnt, s->set[0].counters, 4, cudaMemcpyDeviceToHost);
    out->tiles = cnt;
    s->prof = false;
    s->ev_used = 0;
    s->ev_kind.clear();
    return WV_OK;
}

int wv_launches_per_viewport(const wv_stream *s) {
    if (!s) return WV_ERR_ARG;
    return split_mode(s) ? 5 : 4;
}

int wv_set_decode_mode(wv_stream *s, int mode) {
    if (!s || mode < 0 || mode > 2) return WV_ERR_ARG;
    s->decode_mode = mode;
    return WV_OK;
}

int wv_encode_sizes(const wv_stream_desc *desc, size_t *scratch_bytes, size_t *max_stream_bytes) {
    if (!desc) return WV_ERR_ARG;
    Geom g;
    if (build_geom(*desc, &g) != WV_OK) return WV_ERR_ARG;
    return encode_sizes(g, scratch_bytes, max_stream_bytes);
}

int wv_encode(const wv_stream_desc *desc, const void *const *planes_dev, void *scratch_dev,
              size_t scratch_bytes, void *out, size_t cap, size_t *out_len, void *cuda_stream) {
    if (!desc || !planes_dev || !scratch_dev || !out || !out_len || desc->quant != 0) return WV_ERR_ARG;
    Geom g;
    if (build_geom(*desc, &g) != WV_OK) return WV_ERR_ARG;
    return encode_run(g, planes_dev, scratch_dev, scratch_bytes, out, cap, out_len,
                      (cudaStream_t)cuda_stream);
}

int wv_encode_paper(const wv_stream_desc *desc, const void *const *planes_dev, void *scratch_dev,
                    size_t scratch_bytes, float alpha, float alpha_t, void *out, size_t cap, size_t *out_len,
                    void *cuda_stream) {
    if (!desc || !planes_dev || !scratch_dev || !out || !out_len || desc->quant != 1) return WV_ERR_ARG;
    if (!(alpha >= 0.f) || !(alpha_t >= 0.f) || !isfinite(alpha) || !isfinite(alpha_t)) return WV_ERR_ARG;
    Geom g;
    if (build_geom(*desc, &g) != WV_OK) return WV_ERR_ARG;
    return encode_paper(g, planes_dev, scratch_dev, scratch_bytes, alpha, alpha_t, out, cap, out_len,
                        (cudaStream_t)cuda_stream);
}

}  // extern "C"
