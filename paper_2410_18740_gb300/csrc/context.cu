// Context services: device memory through the caller's allocator (or cudaMalloc),
// grow-only workspace slots, per-kernel-class CUDA-event timing, MPO core upload.
#include <algorithm>
#include <cstring>

#include <map>
#include <mutex>
#include <utility>

#include "vtn_internal.cuh"

namespace vtn {

void* Ctx::dalloc(size_t bytes) {
    if (bytes == 0) bytes = 256;
    bytes = (bytes + 255) & ~size_t(255);
    void* p = nullptr;
    if (has_alloc) {
        p = alloc.alloc(bytes, alloc.user);
        if (!p && drop_digits()) p = alloc.alloc(bytes, alloc.user);
        if (!p) throw Error{VTN_ENOMEM, "device allocation of " + std::to_string(bytes) + " bytes failed"};
    } else {
        cudaError_t e = cudaMalloc(&p, bytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            if (drop_digits()) e = cudaMalloc(&p, bytes);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            throw Error{VTN_ENOMEM, "cudaMalloc(" + std::to_string(bytes) + "): " + cudaGetErrorString(e)};
        }
    }
    return p;
}

void Ctx::dfree(void* p) {
    if (!p) return;
    if (has_alloc) alloc.free(p, alloc.user);
    else cudaFree(p);
}

void set_smem_attr_once(const Ctx& ctx, const void* fn, int bytes) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> done;
    std::lock_guard<std::mutex> lock(mu);
    int& have = done[{fn, ctx.device}];
    if (have >= bytes) return;
    VTN_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    have = bytes;
}

void* Ctx::workspace(int slot, size_t bytes) {
    if ((int)ws.size() < WS_COUNT) ws.resize(WS_COUNT);
    DevBuf& b = ws[slot];
    if (b.bytes < bytes) {
        // the stream may still use the old buffer
        sync();
        dfree(b.p);
        b.p = nullptr;
        b.bytes = 0;
        size_t want = std::max(bytes, size_t(4096));
        b.p = dalloc(want);
        b.bytes = want;
    }
    return b.p;
}

void Ctx::drop(int slot) {
    if (slot >= (int)ws.size() || ws[slot].p == nullptr) return;
    sync();
    dfree(ws[slot].p);
    ws[slot].p = nullptr;
    ws[slot].bytes = 0;
}

bool Ctx::drop_digits() {
    if (digits_busy) return false;
    size_t held = 0;
    for (int s : {WS_OZ_EXP, WS_OZ_A, WS_OZ_B}) {
        if (s < (int)ws.size()) held += ws[s].bytes;
        drop(s);
    }
    return held > 0;
}

double* Ctx::defer_reserve(size_t doubles) {
    if (defer_cap < doubles) {
        sync();
        if (defer_buf) cudaFreeHost(defer_buf);
        defer_buf = nullptr;
        defer_cap = 0;
        const size_t want = std::max(doubles, size_t(4096));
        VTN_CUDA_TRY(cudaMallocHost((void**)&defer_buf, sizeof(double) * want));
        defer_cap = want;
    }
    return defer_buf;
}

int Ctx::tbegin(int cls, double flops) {
    if (!timing) return -1;
    if (pending.size() > 4096 && open_intervals == 0) tflush();
    cudaEvent_t a, bb;
    if (event_pool.size() >= 2) {
        a = event_pool.back(); event_pool.pop_back();
        bb = event_pool.back(); event_pool.pop_back();
    } else {
        VTN_CUDA_TRY(cudaEventCreate(&a));
        VTN_CUDA_TRY(cudaEventCreate(&bb));
    }
    VTN_CUDA_TRY(cudaEventRecord(a, stream));
    pending.push_back(Pending{a, bb, cls, flops});
    ++open_intervals;
    return (int)pending.size() - 1;
}

void Ctx::tend(int idx) {
    if (idx < 0) return;
    VTN_CUDA_TRY(cudaEventRecord(pending[idx].b, stream));
    --open_intervals;
}

void Ctx::tflush() {
    if (pending.empty()) return;
    sync();
    for (auto& p : pending) {
        float ms = 0.f;
        VTN_CUDA_TRY(cudaEventElapsedTime(&ms, p.a, p.b));
        tc[p.cls].launches += 1;
        tc[p.cls].flops += p.flops;
        tc[p.cls].seconds += ms * 1e-3;
        event_pool.push_back(p.a);
        event_pool.push_back(p.b);
    }
    pending.clear();
}

void Ctx::check_dstatus() {
    if (!dstatus) return;
    dstatus_due = false;
    VTN_CUDA_TRY(cudaMemcpyAsync(pinned + 4095, dstatus, sizeof(int), cudaMemcpyDeviceToHost, stream));
    sync();
    int v = 0;
    std::memcpy(&v, pinned + 4095, sizeof(int));
    if (v != 0) {
        VTN_CUDA_TRY(cudaMemsetAsync(dstatus, 0, sizeof(int), stream));
        sync();
        throw Error{VTN_ETIMEOUT, "a bounded device-side wait gave up (tensor-core pipeline)"};
    }
}

void Ctx::check_launch(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error{VTN_ECUDA, std::string(what) + ": " + cudaGetErrorString(e)};
}

// ------------------------------------------------------------------ cores
HostCore core_from_abi(const vtn_core* c, bool copy) {
    VTN_REQUIRE(c != nullptr, "null core");
    VTN_REQUIRE(c->w_left >= 1 && c->w_right >= 1 && c->d >= 1 && c->d <= 16 && c->nnz >= 0,
                "core shape out of range (need w >= 1, 1 <= d <= 16)");
    VTN_REQUIRE(c->nnz == 0 || (c->rows && c->cols && c->ops), "core arrays missing");
    HostCore h;
    h.wl = c->w_left;
    h.wr = c->w_right;
    h.d = c->d;
    const int dd = c->d * c->d, nnz = c->nnz;
    for (int k = 0; k < nnz; ++k)
        VTN_REQUIRE(c->rows[k] >= 0 && c->rows[k] < c->w_left && c->cols[k] >= 0 && c->cols[k] < c->w_right,
                    "core entry channel out of range");
    h.rows.assign(c->rows, c->rows + nnz);
    h.cols.assign(c->cols, c->cols + nnz);
    const cplx* ops = reinterpret_cast<const cplx*>(c->ops);
    if (copy) h.ops.assign(ops, ops + (size_t)nnz * dd);
    else h.ext = ops;
    h.ident.resize(nnz);
    for (int k = 0; k < nnz; ++k) {
        // scaled identity: every entry equals its place in s I (no early exit: the loop vectorises)
        const double* p = c->ops + 2 * (size_t)k * dd;
        const double sr = p[0], si = p[1];
        int bad = 0;
        for (int i = 0; i < 2 * dd; ++i) bad += p[i] != 0.0;
        int diag = 0;
        for (int i = 0; i < c->d; ++i) {
            const double* q = p + 2 * (size_t)i * (c->d + 1);
            bad -= (q[0] != 0.0) + (q[1] != 0.0);
            diag += (q[0] != sr) + (q[1] != si);
        }
        h.ident[k] = bad == 0 && diag == 0 ? 1 : 0;
    }
    return h;
}

void upload_core(Ctx& ctx, const HostCore& hc, DevCore& dc, int what, int slot) {
    dc.wl = hc.wl;
    dc.wr = hc.wr;
    dc.d = hc.d;
    dc.nnz = hc.nnz();
    const int nnz = dc.nnz, d = hc.d;
    // grouped index lists of a subset of the entries: by output column (ptr over wr) or row
    auto group = [&](bool by_col, bool dense_only, std::vector<int>& ptr, std::vector<int>& src,
                     std::vector<int>& op) {
        const int w_out = by_col ? hc.wr : hc.wl;
        ptr.assign(w_out + 1, 0);
        for (int k = 0; k < nnz; ++k)
            if (!dense_only || !hc.ident[k]) ptr[(by_col ? hc.cols[k] : hc.rows[k]) + 1]++;
        for (int b = 0; b < w_out; ++b) ptr[b + 1] += ptr[b];
        src.assign(std::max(ptr[w_out], 0), 0);
        op.assign(src.size(), 0);
        std::vector<int> fill(ptr.begin(), ptr.end() - 1);
        for (int k = 0; k < nnz; ++k) {
            if (dense_only && hc.ident[k]) continue;
            const int o = by_col ? hc.cols[k] : hc.rows[k];
            const int pos = fill[o]++;
            src[pos] = by_col ? hc.rows[k] : hc.cols[k];
            op[pos] = k;
        }
    };
    std::vector<int> col_ptr, col_src, col_op, row_ptr, row_src, row_op;
    group(true, false, col_ptr, col_src, col_op);
    group(false, false, row_ptr, row_src, row_op);
    dc.n_ident = 0;
    dc.n_dense = 0;
    for (int k = 0; k < nnz; ++k) (hc.ident[k] ? dc.n_ident : dc.n_dense)++;
    // a core whose scaled-identity entries fill a large part of the w_l x w_r channel matrix (the
    // collapse core at the centre of the chain) keeps them as a dense matrix C[a][b] as well, and
    // its remaining entries as separate lists: its FP32 mixing is then a channel GEMM plus a
    // sparse pass over the few dense d x d entries
    dc.has_cid = dc.n_ident >= 4 * std::max(hc.wl, hc.wr);
    std::vector<float> cid;
    std::vector<int> dcp, dcs, dco, drp, drs, dro;
    if (dc.has_cid) {
        cid.assign((size_t)2 * hc.wl * hc.wr, 0.f);
        dc.cid_real = true;
        for (int k = 0; k < nnz; ++k) {
            if (!hc.ident[k]) continue;
            const cplx c = hc.op(k)[0];
            const size_t at = (size_t)hc.rows[k] * hc.wr + hc.cols[k];
            cid[2 * at] += (float)c.real();
            cid[2 * at + 1] += (float)c.imag();
            if (c.imag() != 0.0) dc.cid_real = false;
        }
        group(true, true, dcp, dcs, dco);
        group(false, true, drp, drs, dro);
    }
    // spelled-out terms: the groups' entries in order, then the operator's row in order
    std::vector<int> nzp[4];
    std::vector<unsigned> nzs[4];
    std::vector<cplx> nzc[4], cid64;
    const int n_lists = !(what & CORE_F64) ? 0 : dc.has_cid ? 4 : 2;
    for (int l = 0; l < n_lists; ++l) {
        const bool by_col = (l & 1) == 0;
        const std::vector<int>&ptr = l == 0 ? col_ptr : l == 1 ? row_ptr : l == 2 ? dcp : drp,
                              &src = l == 0 ? col_src : l == 1 ? row_src : l == 2 ? dcs : drs,
                              &op = l == 0 ? col_op : l == 1 ? row_op : l == 2 ? dco : dro;
        const int w_out = by_col ? hc.wr : hc.wl;
        nzp[l].reserve((size_t)w_out * d + 1);
        nzs[l].reserve(op.size() * (size_t)d);
        nzc[l].reserve(op.size() * (size_t)d);
        nzp[l].push_back(0);
        auto add = [&](int e, int t, const cplx& c) {
            if (c == cplx(0, 0)) return;
            const unsigned kind = c == cplx(1, 0) ? MIX_ONE : c.imag() == 0.0 ? MIX_REAL : c.real() == 0.0 ? MIX_IMAG : MIX_CPLX;
            nzs[l].push_back((unsigned)(src[e] * d + t) | (kind << 30));
            nzc[l].push_back(c);
        };
        for (int b = 0; b < w_out; ++b)
            for (int sp = 0; sp < d; ++sp) {
                for (int e = ptr[b]; e < ptr[b + 1]; ++e) {
                    const cplx* o = hc.op(op[e]) + (size_t)sp * d;
                    if (hc.ident[op[e]]) add(e, sp, hc.op(op[e])[0]);
                    else
                        for (int t = 0; t < d; ++t) add(e, t, o[t]);
                }
                nzp[l].push_back((int)nzs[l].size());
            }
    }
    if ((what & CORE_F64) && dc.has_cid) {
        cid64.assign((size_t)hc.wl * hc.wr, cplx(0, 0));
        for (int k = 0; k < nnz; ++k)
            if (hc.ident[k]) cid64[(size_t)hc.rows[k] * hc.wr + hc.cols[k]] += hc.op(k)[0];
    }
    // FP32 operators, one scalar for a scaled identity
    const int n_mix = !(what & CORE_F32) ? 0 : dc.has_cid ? 3 : 2;
    std::vector<float> f32;
    std::vector<int> code(n_mix ? nnz : 0);
    for (int k = 0; k < (n_mix ? nnz : 0); ++k) {
        code[k] = (int)f32.size() + (hc.ident[k] ? 1 : 0);  // (floats so far = 2 x complex offset)
        const cplx* o = hc.op(k);
        for (int i = 0; i < (hc.ident[k] ? 1 : d * d); ++i) {
            f32.push_back((float)o[i].real());
            f32.push_back((float)o[i].imag());
        }
    }
    const std::vector<int>* mix[3][2] = {{&col_ptr, &col_src}, {&row_ptr, &row_src}, {&dcp, &dcs}};
    std::vector<int> mix_op[3];
    for (int l = 0; l < n_mix; ++l) {
        const std::vector<int>& op = l == 0 ? col_op : l == 1 ? row_op : dco;
        mix_op[l].resize(op.size());
        for (size_t i = 0; i < op.size(); ++i) mix_op[l][i] = code[op[i]];
    }
    // one block holding everything
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += (std::max(bytes, size_t(1)) + 255) & ~size_t(255); return o; };
    const size_t o_cid = take(sizeof(float) * cid.size()), o_cid64 = take(sizeof(double2) * cid64.size());
    const size_t o_f32 = take(sizeof(float) * f32.size());
    size_t o_p[4], o_s[4], o_c[4], o_m[3][3];
    for (int l = 0; l < n_mix; ++l) {
        o_m[l][0] = take(sizeof(int) * mix[l][0]->size());
        o_m[l][1] = take(sizeof(int) * mix[l][1]->size());
        o_m[l][2] = take(sizeof(int) * mix_op[l].size());
    }
    for (int l = 0; l < n_lists; ++l) {
        o_p[l] = take(sizeof(int) * nzp[l].size());
        o_s[l] = take(sizeof(unsigned) * nzs[l].size());
        o_c[l] = take(sizeof(double2) * nzc[l].size());
    }
    const bool staged = slot >= 0 && off <= Ctx::STAGE * sizeof(double);
    std::vector<unsigned char> owned;
    unsigned char* blob;
    if (staged) {
        blob = (unsigned char*)(ctx.pinned + Ctx::PINNED + (slot == WS_CORE_B ? Ctx::STAGE : 0));
    } else {
        owned.resize(off);
        blob = owned.data();
    }
    auto put = [&](size_t o, const void* p, size_t bytes) {
        if (bytes) std::memcpy(blob + o, p, bytes);
    };
    put(o_cid, cid.data(), sizeof(float) * cid.size());
    put(o_cid64, cid64.data(), sizeof(double2) * cid64.size());
    for (int l = 0; l < n_lists; ++l) {
        put(o_p[l], nzp[l].data(), sizeof(int) * nzp[l].size());
        put(o_s[l], nzs[l].data(), sizeof(unsigned) * nzs[l].size());
        put(o_c[l], nzc[l].data(), sizeof(double2) * nzc[l].size());
    }
    put(o_f32, f32.data(), sizeof(float) * f32.size());
    for (int l = 0; l < n_mix; ++l) {
        put(o_m[l][0], mix[l][0]->data(), sizeof(int) * mix[l][0]->size());
        put(o_m[l][1], mix[l][1]->data(), sizeof(int) * mix[l][1]->size());
        put(o_m[l][2], mix_op[l].data(), sizeof(int) * mix_op[l].size());
    }
    unsigned char* base;
    if (slot >= 0) {
        base = (unsigned char*)ctx.workspace(slot, off);
    } else {
        DevBuf b;
        b.bytes = off;
        b.p = ctx.dalloc(off);
        base = (unsigned char*)b.p;
        dc.bufs.push_back(b);
    }
    VTN_CUDA_TRY(cudaMemcpyAsync(base, blob, off, cudaMemcpyHostToDevice, ctx.stream));
    if (!staged) ctx.sync();  // blob is a local host buffer
    if (dc.has_cid) dc.cid = (float2*)(base + o_cid);
    if (!cid64.empty()) dc.cid64 = (double2*)(base + o_cid64);
    for (int l = 0; l < n_lists; ++l) {
        dc.nz_ptr[l] = (int*)(base + o_p[l]);
        dc.nz_src[l] = (unsigned*)(base + o_s[l]);
        dc.nz_c[l] = (double2*)(base + o_c[l]);
    }
    if (n_mix) dc.ops_f32 = (float2*)(base + o_f32);
    for (int l = 0; l < n_mix; ++l) {
        dc.mix_ptr[l] = (int*)(base + o_m[l][0]);
        dc.mix_src[l] = (int*)(base + o_m[l][1]);
        dc.mix_op[l] = (int*)(base + o_m[l][2]);
    }
}

void free_core(Ctx& ctx, DevCore& dc) {
    for (auto& b : dc.bufs) ctx.dfree(b.p);
    dc.bufs.clear();
}

}  // namespace vtn
