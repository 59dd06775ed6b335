// Shard planner and plan upload (host code).
//
// Sharding format (paper Section 4.1): a tensor's dimensions are combined,
// the result is padded so that the shard count divides it, and shard r is the
// r-th equal slice.  On linear GPU memory combining ALL dimensions is free, so
// the format is "flatten, pad, slice"; each slice (piece) is also rounded up
// to A elements so that 16-byte vectors never straddle two tensors.
// One combined shard is piece r of every tensor, in order (Section 5.2).
#include <stdio.h>
#include <string.h>

#include <new>

#include "ws_internal.h"

static thread_local char g_cuda_err[256] = "";

ws_status ws_cuda_fail(cudaError_t e, const char* what) {
    snprintf(g_cuda_err, sizeof(g_cuda_err), "%s: %s", what, cudaGetErrorString(e));
    return WS_ERR_CUDA;
}

ws_status ws_check_launch(const char* what) {
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? WS_OK : ws_cuda_fail(e, what);
}

extern "C" const char* ws_last_cuda_error(void) { return g_cuda_err; }

extern "C" const char* ws_status_string(ws_status s) {
    switch (s) {
        case WS_OK: return "ok";
        case WS_ERR_INVALID_ARG: return "invalid argument";
        case WS_ERR_ALIGNMENT: return "device pointer not 16-byte aligned";
        case WS_ERR_DTYPE: return "unsupported dtype combination";
        case WS_ERR_WORKSPACE: return "workspace missing or too small";
        case WS_ERR_NOT_UPLOADED: return "plan not uploaded to the device";
        case WS_ERR_CUDA: return "CUDA error";
        case WS_ERR_TOO_LARGE: return "size beyond a fixed limit";
    }
    return "unknown status";
}

// Adafactor's matrix view of every tensor: columns = last dimension, rows = all leading
// dimensions together; fewer than two dimensions: one row, no row accumulator.
static void ws_matrix_views(ws_plan* p, const ws_tensor_desc* descs) {
    p->segaf.resize(p->T);
    p->afchunks.clear();
    long long foff = 0, ioff = 0;
    for (int t = 0; t < p->T; ++t) {
        const ws_tensor_desc& d = descs[t];
        const long long n = p->segs[t].numel;
        WsSegAf a;
        a.foff = foff;
        a.numel = n;
        if (d.ndim >= 2 && n > 0) {
            a.ncol = d.dims[d.ndim - 1];
            a.nrow = n / a.ncol;
        } else {
            a.nrow = 0;
            a.ncol = n;
        }
        foff += a.nrow + a.ncol;
        a.irow = ioff;
        ioff += (a.nrow + 7) / 8 * 8;
        a.icol = ioff;
        ioff += (a.ncol + 7) / 8 * 8;
        p->segaf[t] = a;
        for (long long b = 0; b < a.nrow + a.ncol; b += kWsAfChunk) {
            WsAfChunk c;
            c.begin = b;
            c.count = (int)((a.nrow + a.ncol - b) < kWsAfChunk ? (a.nrow + a.ncol - b) : kWsAfChunk);
            c.seg = t;
            p->afchunks.push_back(c);
        }
    }
    p->F = foff;
    p->Fi = ioff;
}

// Adafactor's blocks (see WsAfItem).  The strips of a row are chosen so that rp rows of tpr threads fill the
// CTA best (a 1200-column matrix: two strips of 75 threads in three rows, 88 % busy, instead of one of 150,
// 59 %).  A block holds up to 65536 elements, fewer where that would leave less than 750 blocks (1.7 waves of
// CTAs): every entry pays a chain of dependent table reads and a barrier.  Measured (Transformer set, 4 copies):
// 16384 elements 1305 us, 32768 1255 us, 65536 1245 us; 22.7 M parameters in ragged tensors, 2 copies: at least
// 3000 blocks 255 us, 1500 194 us, 750 176 us.
template <typename F>
static void ws_af_blocks(const ws_plan* p, F&& emit) {
    long long block = 65536;
    while (block > 1024 && p->N / block < 750) block >>= 1;
    for (int t = 0; t < p->T; ++t) {
        const WsSegAf& a = p->segaf[t];
        if (a.numel <= 0) continue;
        const bool full = a.nrow == 0;
        const long long ncol = full ? (a.numel < 1024 ? a.numel : 1024) : a.ncol;
        const long long nrow = full ? (a.numel + ncol - 1) / ncol : a.nrow;
        const int mode = full ? WS_AF_FULL : ncol % 8 == 0 ? WS_AF_VEC8 : ncol % 4 == 0 ? WS_AF_VEC4 :
                         (4 - ncol % 4) * 8 > ncol ? WS_AF_NARROW : WS_AF_SCALAR;
        const long long W = ws_af_width(mode);
        const long long units = (ncol + W - 1) / W, s0 = (units + 255) / 256;
        long long best_s = s0, best = -1;              // (busy threads of 256) / strips, compared as fractions
        for (long long s = s0; s < s0 + 8 && s <= units; ++s) {
            const long long tpr = (units + s - 1) / s, rows = 256 / tpr < nrow ? 256 / tpr : nrow;
            const long long score = units * rows * 4096 / s;     // (a vector is one row: the fewest strips)
            if (score > best) { best = score; best_s = s; }
        }
        const long long tpr = (units + best_s - 1) / best_s;
        long long rp = 256 / tpr;
        if (rp > nrow) rp = nrow;
        const long long step = rp * (block < 256 * W ? 1 : block / (256 * W));
        for (long long r0 = 0; r0 < nrow; r0 += step)
            for (long long c0 = 0; c0 < ncol; c0 += W * tpr) {
                const long long nc = ncol - c0 < W * tpr ? ncol - c0 : W * tpr;
                const long long nr = nrow - r0 < step ? nrow - r0 : step;
                emit(t, mode, r0, c0, nr, nc, (nc + W - 1) / W, rp);
            }
    }
}

// Block and schedule-entry counts and the floats of kept gradient sums; a tensor beyond the block fields'
// ranges leaves the plan without Adafactor blocks.
static void ws_count_af(ws_plan* p) {
    p->n_afitems = p->n_afsched = p->af_ghat = p->af_rows = p->af_scalar = 0;
    if (p->R > 65535) return;
    long long n = 0, m = 0, g = 0, rows = 0;
    for (const WsSegAf& a : p->segaf) {
        if (a.nrow > 0x7fffffffLL || a.ncol > 0x7fffffffLL) return;
        if (a.nrow > 0) m += (a.nrow + a.ncol + kWsAfChunk - 1) / kWsAfChunk;
        rows += a.nrow;
        if (a.nrow > 0 && a.ncol % 4 != 0) p->af_scalar += a.numel;
    }
    ws_af_blocks(p, [&](int, int mode, long long, long long, long long nr, long long nc, long long tpr, long long) {
        ++n;
        g += (nr * ws_af_kept_row(mode, (int)nc, (int)tpr) + 31) / 32 * 32;
    });
    if (n > 0x0fffffffLL || m > 0x0fffffffLL || g / 32 > 0xffffffffLL) return;
    p->n_afitems = n;
    p->n_afsched = 3 * n + m;
    p->af_ghat = g;
    p->af_rows = rows;
}

// Work items of the one-launch schedule: every run of consecutive positions of one tensor in one shard (a piece;
// in the concatenated layout what lies of the tensor in the shard), cut into items of whole tiles (the partial
// norms are the tiles').  Up to 8192 elements per item - a CTA pays its chain of table reads per item - and fewer
// where that would leave less than 750 items (1.7 waves).  A kernel's pass over an item is 1024 or 2048 elements;
// several tiles share an item only where a pass ends with a tile, or two tiles of 1024 fill one.
template <typename F>
static void ws_lamb_items(const ws_plan* p, F&& emit) {
    const bool concat = p->layout == WS_LAYOUT_CONCAT;
    long long item = kWsItemElems;
    while (item > 1024 && p->N / item < 750) item >>= 1;
    item = (p->K == 1024 || p->K % 2048 == 0) && item > p->K ? item / p->K * p->K : p->K;
    auto cut = [&](int t, int shard, long long pos, long long toff, long long len, long long valid, int tile) {
        for (long long so = 0; so < len; so += item)
            emit(t, shard, pos + so, toff + so, len - so < item ? len - so : item, valid - so, tile + (int)(so / p->K));
    };
    for (int t = 0; t < p->T; ++t) {
        const ws_segment& g = p->segs[t];
        const WsSegTiles st = p->segtiles[t];
        if (!concat) {
            for (int r = 0; r < p->R; ++r) cut(t, r, g.shard_off, r * g.piece, g.piece, g.numel - r * g.piece, st.tile_begin);
            continue;
        }
        for (int k = 0; k < st.tile_count;) {          // a tensor's tiles of one shard are neighbours
            const int k0 = st.tile_begin + k;
            const WsTile& first = p->tiles[k0];
            long long len = 0;
            for (; k < st.tile_count && p->tiles[st.tile_begin + k].shard == first.shard; ++k) len += p->tiles[st.tile_begin + k].len;
            cut(t, first.shard, first.pos, first.poff, len, first.vt, k0);
        }
    }
}

// Plans beyond the item fields' ranges get no schedule (n_items stays 0).
static void ws_count_items(ws_plan* p) {
    p->n_items = 0;
    if (p->R > 65535 || p->S >= (1LL << 47)) return;
    long long n = 0;
    ws_lamb_items(p, [&](int, int, long long, long long, long long, long long, int) { ++n; });
    if (n > 0x3fffffffLL) return;
    p->n_items = n;
}

extern "C" ws_status ws_plan_create(const ws_tensor_desc* descs, int32_t T, int32_t R,
                                    int32_t align_elems, int32_t tile_elems, ws_plan** out) {
    return ws_plan_create_layout(descs, T, R, align_elems, tile_elems, WS_LAYOUT_PER_TENSOR, out);
}

extern "C" int32_t ws_plan_layout(const ws_plan* p) { return p ? p->layout : 0; }

extern "C" ws_status ws_plan_create_layout(const ws_tensor_desc* descs, int32_t T, int32_t R, int32_t align_elems,
                                           int32_t tile_elems, ws_layout layout, ws_plan** out) {
    if (!out) return WS_ERR_INVALID_ARG;
    *out = nullptr;
    if (!descs || T < 1 || R < 1) return WS_ERR_INVALID_ARG;
    if (layout != WS_LAYOUT_PER_TENSOR && layout != WS_LAYOUT_CONCAT) return WS_ERR_INVALID_ARG;
    if (align_elems < 8 || (align_elems & (align_elems - 1)) != 0) return WS_ERR_INVALID_ARG;
    if (tile_elems == 0) {
        // Default: the largest tile that still leaves >= 20000 work items for an all-shard
        // launch.  A CTA reads its tile descriptor before it can issue any data load, so a
        // large tile amortises that latency; small models keep small tiles so that the
        // grid still spreads evenly over the SMs.
        long long total = 0;
        for (int t = 0; t < T; ++t) {
            long long n = 1;
            for (int i = 0; i < descs[t].ndim && i < WS_MAX_DIMS; ++i) n *= (descs[t].dims[i] > 0 ? descs[t].dims[i] : 0);
            total += n;
        }
        // ... and >= 600 items for a single-shard launch (many replicas make tiny shards; a CTA
        // then walks all R gradient slices for its tile, so the grid needs the parallelism).
        tile_elems = 1024;
        if (total / R / 2048 >= 600) tile_elems = 2048;
        while (tile_elems >= 2048 && tile_elems < 8192 && total / (2 * tile_elems) >= 20000 &&
               total / R / (2 * tile_elems) >= 600)
            tile_elems *= 2;
    }
    if (tile_elems < 1024 || tile_elems % 1024 != 0 || tile_elems > (1 << 20)) return WS_ERR_INVALID_ARG;

    ws_plan* p = new (std::nothrow) ws_plan;
    if (!p) return WS_ERR_INVALID_ARG;
    p->T = T;
    p->R = R;
    p->A = align_elems;
    p->K = tile_elems;
    p->layout = layout;
    try {
        p->segs.resize(T);
        p->segtiles.resize(T);
        long long off = 0;
        for (int t = 0; layout == WS_LAYOUT_CONCAT && t < T; ++t) {
            // Concatenated layout (Section 5.2): tensors back to back, each start rounded up to A.
            const ws_tensor_desc& d = descs[t];
            if (d.ndim < 0 || d.ndim > WS_MAX_DIMS) { delete p; return WS_ERR_INVALID_ARG; }
            long long n = 1;
            for (int i = 0; i < d.ndim; ++i) {
                if (d.dims[i] < 0 || (d.dims[i] > 0 && n > (1LL << 46) / d.dims[i])) { delete p; return WS_ERR_INVALID_ARG; }
                n *= d.dims[i];
            }
            p->segs[t].numel = n;
            p->segs[t].piece = 0;
            p->segs[t].shard_off = off;          // start inside the concatenation
            p->N += n;
            p->arena_off.push_back(p->arena_elems);
            p->arena_elems += (n + 7) / 8 * 8;
            off = (off + n + align_elems - 1) / align_elems * align_elems;
        }
        if (layout == WS_LAYOUT_CONCAT) {
            const long long C = off;
            const long long per = (C + R - 1) / R;
            p->S = (per + align_elems - 1) / align_elems * align_elems;
            const long long G = p->S * R;
            // region of tensor t: from its start to the next tensor's start (the alignment gap
            // belongs to it as padding); the last region runs to the end of the last shard
            int t = 0;
            p->shard_tile_begin.assign(R + 1, 0);
            for (int k = 0; k < T; ++k) { p->segtiles[k].tile_begin = 0; p->segtiles[k].tile_count = 0; }
            std::vector<char> seen(T, 0);
            for (int r = 0; r < R; ++r) {
                p->shard_tile_begin[r] = (long long)p->tiles.size();
                long long pos = (long long)r * p->S;            // global position
                const long long end = pos + p->S;
                while (pos < end) {
                    // tensor whose region holds `pos`
                    while (t < T - 1 && p->segs[t + 1].shard_off <= pos) ++t;
                    const long long reg_end = (t < T - 1) ? p->segs[t + 1].shard_off : G;
                    long long stop = reg_end < end ? reg_end : end;
                    long long len = stop - pos;
                    if (len > tile_elems) len = tile_elems;
                    WsTile tl;
                    memset(&tl, 0, sizeof(tl));
                    tl.pos = pos - (long long)r * p->S;
                    tl.poff = pos - p->segs[t].shard_off;
                    tl.vt = p->segs[t].numel - tl.poff;
                    tl.piece = 0;
                    tl.len = (int)len;
                    tl.seg = t;
                    tl.shard = r;
                    if ((long long)p->tiles.size() >= 0x7fffffffLL) { delete p; return WS_ERR_TOO_LARGE; }
                    if (!seen[t]) { seen[t] = 1; p->segtiles[t].tile_begin = (int)p->tiles.size(); }
                    p->segtiles[t].tile_count += 1;
                    p->tiles.push_back(tl);
                    if (tl.len > p->longest) p->longest = tl.len;
                    pos += len;
                }
            }
            p->shard_tile_begin[R] = (long long)p->tiles.size();
            p->ntiles = (long long)p->tiles.size();
            // a tensor without tiles (empty, and no padding region of its own) still names the place
            // in the tile list where its tiles would be, so that a range of tensors maps to a range of tiles
            for (int k = 0; k < T; ++k)
                if (!seen[k])
                    p->segtiles[k].tile_begin = k > 0 ? p->segtiles[k - 1].tile_begin + p->segtiles[k - 1].tile_count : 0;
            ws_matrix_views(p, descs);
            ws_count_items(p);
            ws_count_af(p);
            *out = p;
            return WS_OK;
        }
        for (int t = 0; t < T; ++t) {
            const ws_tensor_desc& d = descs[t];
            if (d.ndim < 0 || d.ndim > WS_MAX_DIMS) { delete p; return WS_ERR_INVALID_ARG; }
            long long n = 1;
            for (int i = 0; i < d.ndim; ++i) {
                if (d.dims[i] < 0 || (d.dims[i] > 0 && n > (1LL << 46) / d.dims[i])) { delete p; return WS_ERR_INVALID_ARG; }
                n *= d.dims[i];   // a zero dimension makes an empty tensor: no piece, no tiles
            }
            long long per = (n + R - 1) / R;
            long long piece = (per + align_elems - 1) / align_elems * align_elems;
            p->segs[t].numel = n;
            p->segs[t].piece = piece;
            p->segs[t].shard_off = off;
            p->N += n;
            p->arena_off.push_back(p->arena_elems);
            p->arena_elems += (n + 7) / 8 * 8;
            // cut the piece into tiles that stay inside it
            long long ntile = (piece + tile_elems - 1) / tile_elems;
            if ((long long)p->tiles.size() + ntile > 0x7fffffffLL) { delete p; return WS_ERR_TOO_LARGE; }
            p->segtiles[t].tile_begin = (int)p->tiles.size();
            p->segtiles[t].tile_count = (int)ntile;
            for (long long i = 0; i < ntile; ++i) {
                WsTile tl;
                memset(&tl, 0, sizeof(tl));
                tl.poff = i * tile_elems;
                tl.pos = off + tl.poff;
                tl.vt = n - tl.poff;
                tl.piece = piece;
                long long len = piece - tl.poff;
                tl.len = (int)(len < tile_elems ? len : tile_elems);
                tl.seg = t;
                p->tiles.push_back(tl);
                if (tl.len > p->longest) p->longest = tl.len;
            }
            off += piece;
        }
        p->S = off;
        p->ntiles = (long long)p->tiles.size();
        ws_matrix_views(p, descs);
        ws_count_items(p);
        ws_count_af(p);
    } catch (...) {
        delete p;
        return WS_ERR_INVALID_ARG;
    }
    *out = p;
    return WS_OK;
}

extern "C" void ws_plan_destroy(ws_plan* plan) { delete plan; }
extern "C" int32_t ws_plan_num_tensors(const ws_plan* p) { return p ? p->T : 0; }
extern "C" int32_t ws_plan_num_shards(const ws_plan* p) { return p ? p->R : 0; }
extern "C" int32_t ws_plan_align(const ws_plan* p) { return p ? p->A : 0; }
extern "C" int64_t ws_plan_shard_elems(const ws_plan* p) { return p ? p->S : 0; }
extern "C" int64_t ws_plan_valid_elems(const ws_plan* p) { return p ? p->N : 0; }
extern "C" int64_t ws_plan_num_tiles(const ws_plan* p) { return p ? p->ntiles : 0; }

extern "C" ws_status ws_plan_segments(const ws_plan* p, const ws_segment** segs, int32_t* T) {
    if (!p || !segs || !T) return WS_ERR_INVALID_ARG;
    *segs = p->segs.data();
    *T = p->T;
    return WS_OK;
}

static size_t round16(size_t x) { return (x + 15) & ~(size_t)15; }

extern "C" size_t ws_plan_device_bytes(const ws_plan* p) {
    if (!p) return 0;
    return round16(p->tiles.size() * sizeof(WsTile)) + round16(p->segtiles.size() * sizeof(WsSegTiles)) +
           round16(p->segaf.size() * sizeof(WsSegAf)) + round16(p->afchunks.size() * sizeof(WsAfChunk));
}

extern "C" int64_t ws_plan_factored_elems(const ws_plan* p) { return p ? p->F : 0; }

extern "C" ws_status ws_plan_factored_layout(const ws_plan* p, int64_t* layout) {
    if (!p || !layout) return WS_ERR_INVALID_ARG;
    for (int t = 0; t < p->T; ++t) {
        const WsSegAf& a = p->segaf[t];
        layout[3 * t] = a.foff;
        layout[3 * t + 1] = a.nrow > 0 ? a.nrow : a.ncol;
        layout[3 * t + 2] = a.nrow > 0 ? a.ncol : 0;
    }
    return WS_OK;
}

// Copies `n` tables to their offsets in one device buffer.  Small plans: as one image, one copy (every
// cudaMemcpyAsync from pageable memory costs the host some 10 us); from 128 KB on gathering the image costs more.
// The image and the tables are the plan's: under stream capture the copy becomes a node that reads them at replay.
static ws_status upload_image(char* dev, const void* const* src, const size_t* nb, const size_t* off, int n, size_t total,
                              std::vector<char>& image, cudaStream_t st, const char* what) {
    cudaError_t e = cudaSuccess;
    if (total <= (128u << 10)) {
        if (image.empty()) {                 // (a plan's tables never change once they are built)
            try {
                image.resize(total);
            } catch (...) {
                return WS_ERR_INVALID_ARG;
            }
            for (int i = 0; i < n; ++i)
                if (nb[i]) memcpy(image.data() + off[i], src[i], nb[i]);
        }
        if (total) e = cudaMemcpyAsync(dev, image.data(), total, cudaMemcpyHostToDevice, st);
    } else {
        for (int i = 0; i < n && e == cudaSuccess; ++i)
            if (nb[i]) e = cudaMemcpyAsync(dev + off[i], src[i], nb[i], cudaMemcpyHostToDevice, st);
    }
    return e == cudaSuccess ? WS_OK : ws_cuda_fail(e, what);
}

extern "C" ws_status ws_plan_upload(ws_plan* p, void* dev_buf, size_t bytes, void* stream) {
    if (!p || !dev_buf) return WS_ERR_INVALID_ARG;
    if (!ws_aligned16(dev_buf)) return WS_ERR_ALIGNMENT;
    if (bytes < ws_plan_device_bytes(p)) return WS_ERR_WORKSPACE;
    char* base = (char*)dev_buf;
    size_t o[4], at = 0;
    const size_t nb[4] = {p->tiles.size() * sizeof(WsTile), p->segtiles.size() * sizeof(WsSegTiles),
                          p->segaf.size() * sizeof(WsSegAf), p->afchunks.size() * sizeof(WsAfChunk)};
    const void* src[4] = {p->tiles.data(), p->segtiles.data(), p->segaf.data(), p->afchunks.data()};
    for (int i = 0; i < 4; ++i) { o[i] = at; at += round16(nb[i]); }
    const ws_status s = upload_image(base, src, nb, o, 4, at, p->table_image, (cudaStream_t)stream, "ws_plan_upload");
    if (s != WS_OK) return s;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        p->sms = 148;
    p->d_tiles = (const WsTile*)(base + o[0]);
    p->d_segtiles = (const WsSegTiles*)(base + o[1]);
    p->d_segaf = (const WsSegAf*)(base + o[2]);
    p->d_afchunks = (const WsAfChunk*)(base + o[3]);
    return WS_OK;
}

WsLambWs ws_lamb_layout(const ws_plan* p, void* workspace) {
    WsLambWs L;
    char* b = (char*)workspace;
    size_t o = 0;
    L.rho = (float*)(b + o);
    o = round16(o + sizeof(float) * (size_t)p->T);
    L.norms = (double*)(b + o);
    o = round16(o + sizeof(double) * 2 * (size_t)p->T);
    L.partials = (float2*)(b + o);
    o = round16(o + sizeof(float2) * (size_t)(p->layout == WS_LAYOUT_CONCAT ? 1 : p->R) * (size_t)p->ntiles);
    const size_t sync0 = o;
    L.count = (int*)(b + o);
    o = (o + sizeof(int) * (size_t)p->T + 7) & ~(size_t)7;
    L.flag = (unsigned long long*)(b + o);
    o += sizeof(unsigned long long) * (size_t)p->T;
    L.ticket = (unsigned long long*)(b + o);
    o += sizeof(unsigned long long);
    L.status = (int*)(b + o);
    o = round16(o + sizeof(int));
    L.sync_bytes = o - sync0;
    L.bytes = o;
    o = (o + 255) & ~(size_t)255;
    L.ghat = (float*)(b + o);
    L.bytes_lars = o + sizeof(float) * (size_t)p->R * (size_t)p->S;
    // (the one-kernel Adafactor keeps the sums block by block, which may be more than [R][S] by an eighth and by
    // less than 128 bytes a block)
    const size_t ghat_af = (size_t)p->af_ghat > (size_t)p->R * (size_t)p->S ? (size_t)p->af_ghat : (size_t)p->R * (size_t)p->S;
    o = ((size_t)((char*)L.ghat - b) + sizeof(float) * ghat_af + 255) & ~(size_t)255;
    L.acc = (float*)(b + o);
    const size_t acc0 = o;
    o = (o + sizeof(float) * (size_t)p->Fi + 15) & ~(size_t)15;
    L.rsum = (double*)(b + o);
    o += sizeof(double) * (size_t)p->T;
    L.acc_bytes = o - acc0;
    const size_t T = (size_t)p->T;
    L.af_flagm = (unsigned long long*)(b + o);
    L.af_flag2 = L.af_flagm + T;
    L.af_ticket = L.af_flag2 + T;
    o += sizeof(unsigned long long) * (2 * T + 1);
    L.af_count1 = (int*)(b + o);
    L.af_countm = L.af_count1 + T;
    L.af_count2 = L.af_countm + T;
    o = round16(o + sizeof(int) * 3 * T);
    L.af_sync_bytes = o - acc0;
    L.af_ipart = (double2*)(b + o);
    o += sizeof(double2) * (size_t)p->n_afitems;
    L.af_rfac = (double*)(b + o);
    o += sizeof(double) * (size_t)p->af_rows;
    o = (o + 255) & ~(size_t)255;
    L.fac = (float*)(b + o);
    o = (o + sizeof(float) * (size_t)p->Fi + 255) & ~(size_t)255;
    L.alpha = (float*)(b + o);
    L.bytes_af = o + sizeof(float) * (size_t)p->T;
    return L;
}

extern "C" ws_status ws_workspace_partials(const ws_plan* p, size_t* offset_bytes, size_t* row_bytes) {
    if (!p || !offset_bytes || !row_bytes || p->layout != WS_LAYOUT_PER_TENSOR) return WS_ERR_INVALID_ARG;
    const WsLambWs L = ws_lamb_layout(p, nullptr);
    *offset_bytes = (size_t)((char*)L.partials - (char*)nullptr);
    *row_bytes = sizeof(float2) * (size_t)p->ntiles;
    return WS_OK;
}

extern "C" ws_status ws_workspace_adafactor_sums(const ws_plan* p, size_t* offset_bytes, size_t* bytes) {
    if (!p || !offset_bytes || !bytes) return WS_ERR_INVALID_ARG;
    const WsLambWs L = ws_lamb_layout(p, nullptr);
    *offset_bytes = (size_t)((char*)L.acc - (char*)nullptr);
    *bytes = sizeof(float) * (size_t)p->Fi;
    return WS_OK;
}

extern "C" size_t ws_workspace_bytes(const ws_plan* p, ws_opt opt) {
    if (!p) return 0;
    if (opt == WS_LAMB) return ws_lamb_layout(p, nullptr).bytes;
    if (opt == WS_LARS) return ws_lamb_layout(p, nullptr).bytes_lars;
    if (opt == WS_ADAFACTOR) return ws_lamb_layout(p, nullptr).bytes_af;
    return 0;
}

// ------------------------------------------------------ one-launch schedule ---
// Order of execution for the one-kernel LAMB / LARS update.  Tensors are taken in groups of a few
// megabytes of state; a group's phase-2 items follow its phase-1 items at a distance of at least
// kLag schedule entries (by then every CTA that worked on the group's phase 1 has finished and the
// tensors' ratios are known, so no CTA waits), interleaved one to one with the phase-1 items of the
// following groups: phase 2 then reads w, m', v' out of L2 while phase 1 of the next tensors streams
// from DRAM, and each operand crosses HBM once (Section 2.2).  When more than kLag eligible phase-2
// items are waiting (a tensor larger than L2 has just finished) they run first.
namespace {
constexpr long long kGroupBytes = 6LL << 20;    // state bytes (12 per element) that close a group
constexpr int kLag = 512;

void ws_build_schedule(ws_plan* p) {
    const int T = p->T;
    p->items.clear();
    p->items.reserve((size_t)p->n_items);
    p->itemsegs.assign(T, WsItemSeg{0, 0, 0, 0});
    for (int t = 0; t < T; ++t) {
        p->itemsegs[t].tile_begin = p->segtiles[t].tile_begin;
        p->itemsegs[t].tile_count = p->segtiles[t].tile_count;
    }
    std::vector<long long> seg_bytes(T, 0);
    ws_lamb_items(p, [&](int t, int shard, long long pos, long long toff, long long len, long long valid, int tile) {
        WsItem it;
        it.pos_shard = (unsigned long long)pos << 16 | (unsigned)shard;
        it.toff = toff;
        it.seg = t;
        it.nvalid = (int)(valid < 0 ? 0 : (valid > len ? len : valid));
        it.len = (int)len;
        it.tile = tile;
        p->items.push_back(it);
        ++p->itemsegs[t].count;
        seg_bytes[t] += 12LL * len;
    });
    for (int t = 1; t < T; ++t) p->itemsegs[t].first = p->itemsegs[t - 1].first + p->itemsegs[t - 1].count;
    // groups of consecutive tensors
    struct Group { int first, end; };     // item range
    std::vector<Group> groups;
    {
        long long acc = 0;
        int gfirst = 0;
        for (int t = 0; t < T; ++t) {
            acc += seg_bytes[t];
            const bool last = t == T - 1;
            if (acc >= kGroupBytes || last) {
                const int gend = p->itemsegs[t].first + p->itemsegs[t].count;
                if (gend > gfirst) groups.push_back(Group{gfirst, gend});
                gfirst = gend;
                acc = 0;
            }
        }
    }
    // merge the phase-1 stream and the phase-2 stream
    const long long n = (long long)p->items.size();
    p->sched.clear();
    p->sched.reserve((size_t)(2 * n));
    const int G = (int)groups.size();
    std::vector<long long> p1_done_at(G, -1);     // schedule position of each group's last phase-1 item
    int ag = 0, eg = 0;                           // group of the next phase-1 item; first group not yet eligible
    long long ai = 0, bi = 0;                     // next phase-1 / phase-2 item
    long long eligible = 0;                       // phase-2 items of groups whose phase 1 ended >= kLag entries ago
    int last_kind = 1;
    // phase 2 walks every group back to front: the items phase 1 wrote last are the ones most likely to be
    // in L2 still, and a group larger than the L2 then keeps its tail instead of nothing (reading it front
    // to back would evict each line just before its turn)
    std::vector<unsigned> p2item((size_t)n);
    for (const Group& g : groups)
        for (int i = g.first; i < g.end; ++i) p2item[(size_t)i] = (unsigned)(g.end - 1 - (i - g.first));
    while (bi < n) {
        const long long pos = (long long)p->sched.size();
        while (eg < ag && pos - p1_done_at[eg] >= kLag) {
            eligible += groups[eg].end - groups[eg].first;
            ++eg;
        }
        const long long backlog = eligible - bi;
        const bool may2 = backlog > 0;
        if (ai < n && !(may2 && (last_kind == 0 || backlog > kLag))) {
            p->sched.push_back((unsigned)(ai << 1));
            last_kind = 0;
            if (++ai == groups[ag].end) {
                p1_done_at[ag] = pos;
                ++ag;
            }
        } else {
            // (at the very end the last groups' phase 2 follows their phase 1 directly: the scheduling
            // warps then wait for the ratios, a few microseconds once per launch)
            p->sched.push_back((p2item[(size_t)bi] << 1) | 1u);
            last_kind = 1;
            ++bi;
            if (!may2) eligible = bi;             // keep the backlog arithmetic consistent in the tail
        }
    }
}

// Adafactor: sums (P1) -> moments of every 1024-entry chunk (M) -> U^2 (P2) -> apply (P3).  Groups of tensors
// as above; a phase of a group starts at least kLag entries after its previous one ended, and the phases of
// different groups alternate, so that P1 (and P2's weights) stream from DRAM while the others work from L2.
// P2 walks a group back to front and P3 front to back, each starting with what the one before touched last.
constexpr long long kAfGroupElems = 512 << 10;

void ws_build_af_schedule(ws_plan* p) {
    const int T = p->T;
    std::vector<WsAfItem> items;
    items.reserve((size_t)p->n_afitems);
    p->aftensors.resize(T);
    long long rows = 0;
    for (int t = 0; t < T; ++t) {
        const WsSegAf& a = p->segaf[t];
        WsAfTensor& d = p->aftensors[t];
        memset(&d, 0, sizeof(d));
        d.numel = a.numel; d.ncol = a.ncol; d.nrow = a.nrow;
        d.foff = a.foff; d.irow = a.irow; d.icol = a.icol;
        d.rfac = rows;
        rows += a.nrow;
        d.piece = p->layout == WS_LAYOUT_CONCAT ? (1LL << 62) : p->segs[t].piece;
        d.off = p->segs[t].shard_off;
        d.pad_end = (t + 1 < T ? p->segs[t + 1].shard_off : (long long)p->R * p->S) - d.off;
        d.chunk_count = a.nrow > 0 ? (int)((a.nrow + a.ncol + kWsAfChunk - 1) / kWsAfChunk) : 0;
        d.mode = a.nrow > 0 ? WS_AF_VEC4 : WS_AF_FULL;
        if (d.mode == WS_AF_FULL) d.ncol = a.numel < 1024 ? a.numel : 1024;
    }
    long long goff = 0;
    ws_af_blocks(p, [&](int t, int mode, long long r0, long long c0, long long nr, long long nc, long long tpr, long long rp) {
        WsAfTensor& d = p->aftensors[t];
        if (d.item_count++ == 0) d.item_first = (int)items.size();
        d.mode = mode;
        WsAfItem it;
        memset(&it, 0, sizeof(it));
        it.seg = t;
        it.row0 = (int)r0; it.col0 = (int)c0;
        it.nr = (unsigned short)nr; it.nc = (unsigned short)nc;
        it.tpr = (unsigned short)tpr; it.rp = (unsigned short)rp;
        it.goff32 = (unsigned)goff;
        it.item = (unsigned)items.size();
        goff += (nr * ws_af_kept_row(mode, (int)nc, (int)tpr) + 31) / 32;
        items.push_back(it);
    });
    // groups of consecutive tensors; a group's chunks are consecutive too, once the unfactored tensors' are left out
    struct Group { int i0, i1, m0, m1; };
    std::vector<Group> groups;
    std::vector<int> chunks;
    chunks.reserve((size_t)(p->n_afsched - 3 * p->n_afitems));
    {
        Group g{0, 0, 0, 0};
        long long acc = 0;
        int c = 0;
        for (int t = 0; t < T; ++t) {
            const WsAfTensor& d = p->aftensors[t];
            for (int k = 0; k < d.chunk_count; ++k) chunks.push_back(c + k);
            c += (int)((p->segaf[t].nrow + p->segaf[t].ncol + kWsAfChunk - 1) / kWsAfChunk);
            if (d.item_count == 0) continue;
            g.i1 = d.item_first + d.item_count;
            g.m1 = (int)chunks.size();
            acc += d.numel;
            if (acc >= kAfGroupElems) {
                groups.push_back(g);
                g = Group{g.i1, g.i1, g.m1, g.m1};
                acc = 0;
            }
        }
        if (g.i1 > g.i0) groups.push_back(g);
    }
    std::vector<WsAfItem>& out = p->afsched;
    out.resize((size_t)p->n_afsched);
    const int G = (int)groups.size();
    constexpr long long kNever = 1LL << 62;
    // phase ph works on group next[ph], of which `left` entries are to come, and may go on from position from[ph]
    // (kNever: the phase before has not ended the group yet)
    struct Phase { int next; int left; long long from; } ph[4];
    std::vector<long long> done[4];                   // position after a group's last entry of the phase
    for (auto& d : done) d.assign(G, kNever);
    auto size_of = [&](int c, int g) { return c == 1 ? groups[g].m1 - groups[g].m0 : groups[g].i1 - groups[g].i0; };
    auto open = [&](int c) {                          // phase c turns to group next[c]
        Phase& f = ph[c];
        if (f.next >= G) { f.from = kNever; return; }
        f.left = size_of(c, f.next);
        f.from = c == 0 ? 0 : done[c - 1][f.next] == kNever ? kNever : done[c - 1][f.next] + kLag - 1;
    };
    for (int c = 0; c < 4; ++c) { ph[c].next = 0; open(c); }
    long long pos = 0;
    auto emit = [&](int c) {
        Phase& f = ph[c];
        const Group& g = groups[f.next];
        if (f.left > 0) {
            WsAfItem& rec = out[(size_t)pos++];
            if (c == 1) {
                const WsAfChunk& k = p->afchunks[(size_t)chunks[(size_t)(g.m1 - f.left)]];
                memset(&rec, 0, sizeof(rec));
                rec.seg = k.seg;
                rec.row0 = (int)(unsigned)((unsigned long long)k.begin & 0xffffffffu);
                rec.col0 = (int)(k.begin >> 32);
                rec.goff32 = (unsigned)k.count;
            } else {
                rec = items[(size_t)(c == 2 ? g.i0 + f.left - 1 : g.i1 - f.left)];
            }
            rec.phase = c;
            --f.left;
            f.from = 0;
        }
        if (f.left > 0) return;
        const int g_done = f.next++;
        done[c][g_done] = pos;
        open(c);
        if (c < 3 && ph[c + 1].next == g_done) open(c + 1);
    };
    int last = 3;
    while (ph[3].next < G) {
        int c = -1;
        if (ph[1].from <= pos) {
            c = 1;
        } else {
            for (int k = 1; k <= 4 && c < 0; ++k) {
                const int t = (last + k) & 3;
                if (t != 1 && ph[t].from <= pos) c = t;
            }
        }
        for (int t = 1; t < 4 && c < 0; ++t)           // the tail: nothing is far enough behind
            if (ph[t].from != kNever) c = t;
        emit(c);
        if (c != 1) last = c;
    }
}

size_t af_schedule_bytes(const ws_plan* p) {
    if (p->n_afitems <= 0) return 0;
    return round16((size_t)p->T * sizeof(WsAfTensor)) + (size_t)p->n_afsched * sizeof(WsAfItem);
}
size_t lamb_schedule_bytes(const ws_plan* p) {
    return round16((size_t)p->n_items * sizeof(WsItem)) + round16((size_t)p->T * sizeof(WsItemSeg)) +
           round16((size_t)p->n_items * 2 * sizeof(unsigned));
}
size_t schedule_bytes(const ws_plan* p) { return lamb_schedule_bytes(p) + af_schedule_bytes(p); }
}  // namespace

extern "C" size_t ws_plan_schedule_bytes(const ws_plan* p) {
    if (!p || p->n_items <= 0) return 0;
    return schedule_bytes(p);
}

extern "C" ws_status ws_plan_upload_schedule(ws_plan* p, void* dev_buf, size_t bytes, void* stream) {
    if (!p || !dev_buf) return WS_ERR_INVALID_ARG;
    if (p->n_items <= 0) return WS_ERR_TOO_LARGE;
    if (!ws_aligned16(dev_buf)) return WS_ERR_ALIGNMENT;
    if (bytes < schedule_bytes(p)) return WS_ERR_WORKSPACE;
    try {
        if (p->sched.empty()) ws_build_schedule(p);
        if (p->afsched.empty() && p->n_afitems > 0) ws_build_af_schedule(p);
    } catch (...) {
        return WS_ERR_INVALID_ARG;
    }
    if ((long long)p->items.size() != p->n_items || (long long)p->afsched.size() != p->n_afsched) return WS_ERR_INVALID_ARG;
    char* base = (char*)dev_buf;
    const bool af = p->n_afitems > 0;
    size_t o[5], at = 0;
    const size_t nb[5] = {p->items.size() * sizeof(WsItem), p->itemsegs.size() * sizeof(WsItemSeg),
                          p->sched.size() * sizeof(unsigned), p->aftensors.size() * sizeof(WsAfTensor),
                          p->afsched.size() * sizeof(WsAfItem)};
    const void* src[5] = {p->items.data(), p->itemsegs.data(), p->sched.data(), p->aftensors.data(), p->afsched.data()};
    for (int i = 0; i < (af ? 5 : 3); ++i) { o[i] = at; at += round16(nb[i]); }
    const ws_status s = upload_image(base, src, nb, o, af ? 5 : 3, at, p->sched_image, (cudaStream_t)stream, "ws_plan_upload_schedule");
    if (s != WS_OK) return s;
    p->d_items = (const WsItem*)(base + o[0]);
    p->d_itemsegs = (const WsItemSeg*)(base + o[1]);
    p->d_sched = (const unsigned*)(base + o[2]);
    if (af) {
        p->d_aftensors = (const WsAfTensor*)(base + o[3]);
        p->d_afsched = (const WsAfItem*)(base + o[4]);
    }
    return WS_OK;
}

extern "C" ws_status ws_plan_schedule_view(ws_plan* p, const uint32_t** order, int64_t* n_entries) {
    if (!p || !order || !n_entries) return WS_ERR_INVALID_ARG;
    if (p->n_items <= 0) return WS_ERR_TOO_LARGE;
    try {
        if (p->sched.empty()) ws_build_schedule(p);
    } catch (...) {
        return WS_ERR_INVALID_ARG;
    }
    *order = p->sched.data();
    *n_entries = (int64_t)p->sched.size();
    return WS_OK;
}

extern "C" ws_status ws_plan_schedule_item(ws_plan* p, int64_t item, ws_sched_item* out) {
    if (!p || !out) return WS_ERR_INVALID_ARG;
    if (p->n_items <= 0) return WS_ERR_TOO_LARGE;
    try {
        if (p->sched.empty()) ws_build_schedule(p);
    } catch (...) {
        return WS_ERR_INVALID_ARG;
    }
    if (item < 0 || item >= p->n_items) return WS_ERR_INVALID_ARG;
    const WsItem& it = p->items[(size_t)item];
    out->tensor = it.seg;
    out->shard = (int32_t)(it.pos_shard & 0xffffu);
    out->pos = (int64_t)(it.pos_shard >> 16);
    out->tensor_off = it.toff;
    out->len = it.len;
    out->nvalid = it.nvalid;
    return WS_OK;
}

extern "C" ws_status ws_workspace_sync_status(const ws_plan* p, size_t* offset_bytes) {
    if (!p || !offset_bytes) return WS_ERR_INVALID_ARG;
    const WsLambWs L = ws_lamb_layout(p, nullptr);
    *offset_bytes = (size_t)((char*)L.status - (char*)nullptr);
    return WS_OK;
}
