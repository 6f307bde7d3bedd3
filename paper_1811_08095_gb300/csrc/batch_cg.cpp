// Slot-based batched CG (see batch_cg.h).
#include "batch_cg.h"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

namespace odwf {

Lk link_format(const odwf_solve_params& prm) {
    if (prm.link_prec == ODWF_F16) return Lk::H12;
    return prm.link_recon == 18 ? Lk::F18 : Lk::F12;
}

void CgHost::drop_graphs() {
    for (auto& kv : graphs)
        if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
    graphs.clear();
}

CgHost::~CgHost() {
    drop_graphs();
    for (cudaEvent_t e : ev_rel) cudaEventDestroy(e);
    for (cudaStream_t q : {s_rel, s_solve})
        if (q) {
            cudaStreamSynchronize(q);
            cudaStreamDestroy(q);
        }
    for (cudaEvent_t e : {ev_sync, ev_solve})
        if (e) cudaEventDestroy(e);
    if (pinned) cudaFreeHost(pinned);
}

BatchCG::~BatchCG() {
    if (!H) return;
    if (!idle) cudaDeviceSynchronize();  // an error left copies to the pinned memory in flight
    else if (s_rel) cudaStreamSynchronize(s_rel);
    H->busy = false;
}

template <>
HopParams<double> BatchCG::params<double>(int p_out) const {
    auto P = E->hop_params<double>(p_out, r_dev);
    P.st = st;
    P.partials = partials;
    P.part_stride = nblk;
    P.counters = counters;
    return P;
}

template <>
HopParams<float> BatchCG::params<float>(int p_out) const {
    auto P = E->hop_params<float>(p_out, r_dev);
    P.links = v2 ? E->links_site[(int)lk] : E->links_of(lk);
    P.st = st;
    P.partials = partials;
    P.part_stride = nblk;
    P.counters = counters;
    return P;
}

int BatchCG::init(Engine* e, int capacity, const odwf_solve_params& prm, cudaStream_t s, int update_prio_drop) {
    E = e;
    cap = capacity;
    mixed = prm.prec != ODWF_F64;
    low = (Sp)prm.prec;
    lk = link_format(prm);
    delta = prm.delta > 0 ? prm.delta : 0.01;
    tol = prm.tol;
    max_iter = prm.max_iter;
    int rc = 0;
    const int nrb = mixed ? 1 : cap;  // mixed: R64 and B64 are shared by all systems
    if ((rc = E->alloc_half("cg.X64", Sp::F64, cap, &X64)) || (rc = E->alloc_half("cg.R64", Sp::F64, nrb, &R64)) ||
        (rc = E->alloc_half("cg.B64", Sp::F64, nrb, &B64)))
        return rc;
    if (!mixed) {
        if ((rc = E->alloc_half("cg.P64", Sp::F64, cap, &P64)) || (rc = E->alloc_half("cg.A64", Sp::FX, cap, &A64)) ||
            (rc = E->alloc_half("cg.C64", Sp::FX, cap, &C64)))
            return rc;
    } else {
        const std::string tag = "cg.lo" + std::to_string((int)low);
        if ((rc = E->alloc_half("cg.Rin", Sp::F32, cap, &Rin)) || (rc = E->alloc_half("cg.Xin", Sp::F32, cap, &Xin)) ||
            (rc = E->alloc_half(tag + ".P", low, cap, &Pl)) || (rc = E->alloc_half(tag + ".T", low, cap, &Tl)) ||
            (rc = E->alloc_half(tag + ".A", low, cap, &Al)) || (rc = E->alloc_half(tag + ".C", low, cap, &Cl)) ||
            (rc = E->alloc_half("cg.A1", Sp::FX, 1, &A1)) || (rc = E->alloc_half("cg.C1", Sp::FX, 1, &C1)))
            return rc;
        if ((rc = E->ensure_links(lk, s))) return rc;
        v2 = hop2_supported(E->ns, low, E->vh());
        if (lk == Lk::H12 && !v2) return fail(ODWF_EINVAL, "solve: FP16 links need Ns = 8 or 16");
        if (v2 && (rc = E->alloc_half(tag + ".X", low, cap, &Chil))) return rc;
        if (v2 && (rc = E->ensure_site_links(lk, s))) return rc;
    }
    st = (SysState*)E->get_ws("cg.state", sizeof(SysState) * cap, &rc);
    if (rc) return rc;
    r_dev = (double*)E->get_ws("cg.r", sizeof(double) * cap, &rc);
    if (rc) return rc;
    // one partial per block of a reducing launch and system: sized for the smallest reducing
    // block (64 threads, one 5D site each), so every kernel's grid fits
    nblk = blocks_for(E->sites5(), kMinReduceBlock);
    partials = (double*)E->get_ws("cg.partials", sizeof(double) * (size_t)(nblk + reduce_groups(nblk)) * cap, &rc);
    if (rc) return rc;
    const size_t cbytes = sizeof(unsigned) * (size_t)(reduce_groups(nblk) + 1) * cap;
    counters = (unsigned*)E->get_ws("cg.counters", cbytes, &rc);
    if (rc) return rc;
    ODWF_CK(cudaMemsetAsync(counters, 0, cbytes, s));
    if (!E->cg_host.busy) {
        H = &E->cg_host;
    } else {
        own = std::make_unique<CgHost>();
        H = own.get();
    }
    H->busy = true;
    // pinned: state mirror [cap], initial-state staging [cap], r staging [cap]
    const size_t pb = 2 * sizeof(SysState) * cap + sizeof(double) * cap;
    if (H->pinned_bytes < pb) {
        if (H->pinned) cudaFreeHost(H->pinned);
        H->pinned = nullptr;
        H->pinned_bytes = 0;
        if (cudaMallocHost(&H->pinned, pb) != cudaSuccess) {
            cudaGetLastError();
            H->pinned = nullptr;
            return fail(ODWF_ENOMEM, "pinned host allocation failed");
        }
        H->pinned_bytes = pb;
    }
    st_host = (SysState*)H->pinned;
    std::memset(st_host, 0, sizeof(SysState) * cap);
    for (int i = 0; i < cap; ++i) st_host[i].status = kIdle;
    ODWF_CK(cudaMemcpyAsync(st, st_host, sizeof(SysState) * cap, cudaMemcpyHostToDevice, s));
    ODWF_CK(cudaStreamSynchronize(s));
    n_reliable.assign(cap, 0);
    upd.assign(cap, 0);
    int prio = 0, least = 0, greatest = 0;
    ODWF_CK(cudaStreamGetPriority(s, &prio));
    ODWF_CK(cudaDeviceGetStreamPriorityRange(&least, &greatest));
    const int rel_prio = std::min(least, prio + update_prio_drop);
    if (H->s_rel && H->s_rel_prio != rel_prio) {
        ODWF_CK(cudaStreamDestroy(H->s_rel));
        H->s_rel = nullptr;
    }
    if (!H->s_rel) ODWF_CK(cudaStreamCreateWithPriority(&H->s_rel, cudaStreamNonBlocking, rel_prio));
    H->s_rel_prio = rel_prio;
    s_rel = H->s_rel;
    if (!H->ev_sync) ODWF_CK(cudaEventCreateWithFlags(&H->ev_sync, cudaEventDisableTiming));
    ev_sync = H->ev_sync;
    while ((int)H->ev_rel.size() < cap) {
        cudaEvent_t e = nullptr;
        ODWF_CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        H->ev_rel.push_back(e);
    }
    ev_rel.assign(H->ev_rel.begin(), H->ev_rel.begin() + cap);
    // what the iteration's kernels are launched with, besides the slot range and the iteration count
    const void* bufs[] = {X64.data, R64.data, P64.data, A64.data, C64.data, Rin.data, Xin.data, Pl.data, Tl.data,
                          Al.data, Cl.data, Chil.data, A64.norm, C64.norm, Pl.norm, Tl.norm, Al.norm, Cl.norm,
                          Chil.norm, st, r_dev, partials, counters, E->links_fx, E->nbr,
                          mixed ? E->links_of(lk) : nullptr, v2 ? E->links_site[(int)lk] : nullptr};
    const int fmt[] = {(int)low, (int)lk, mixed, v2, cap, nblk};
    graph_key.assign((const char*)bufs, sizeof(bufs));
    graph_key.append((const char*)fmt, sizeof(fmt));
    bsrc.assign(cap, nullptr);
    active.assign(cap, 0);
    mq.assign(cap, 0.0);
    slot_tol.assign(cap, tol);
    // profiler classes with their algorithmic bytes (each field read or written once)
    const double n5 = (double)E->sites5();
    const double sp = !mixed ? 192.0 : (low == Sp::F32 ? 96.0 : 52.0);  // FP16/BF16: 48 + 4-byte scale
    const double acc = mixed ? 96.0 : 192.0;                              // r, x
    const double links = 8.0 * (double)E->vh() * (!mixed ? 144.0 : lk == Lk::F12 ? 48.0 : lk == Lk::H12 ? 24.0 : 72.0);
    const char* lowname[] = {"f64", "f32", "f16", "bf16"};
    const std::string pre = !mixed ? std::string("f64") :
        std::string("mixed.") + lowname[(int)low] + (lk == Lk::F12 ? ".l12" : lk == Lk::H12 ? ".lh12" : ".l18");
    if (v2) {
        const std::string p2 = pre + ".v2";
        const char* kn[5] = {".K1_chi_minv", ".K2_schur_norm_mdinv", ".K3_dag_minvdag", ".K4_normal_cg", ".P_update_chi"};
        const double ksys[5] = {n5 * 2 * sp, n5 * 3 * sp, n5 * 2 * sp, n5 * (3 * sp + 4 * acc), n5 * (acc + 3 * sp)};
        for (int k = 0; k < 5; ++k) {
            kname[k] = p2 + kn[k];
            kbytes_sys[k] = ksys[k];
            kbytes_launch[k] = k < 4 ? links : 0.0;
            pcls[k] = prof_class(kname[k], kbytes_sys[k], kbytes_launch[k]);
        }
        pcls[5] = prof_class(p2 + ".beta_sum", 0.0, 8.0 * hop_blocks(E->ns, low, 4, E->vh(), 1));
    } else {
    pcls[0] = prof_class(pre + ".K1_minv", n5 * 2 * sp, links);
    pcls[1] = prof_class(pre + ".K2_schur_norm_mdinv", n5 * 3 * sp, links);
    pcls[2] = prof_class(pre + ".K3_dag_minvdag", n5 * 2 * sp, links);
    pcls[3] = prof_class(pre + ".K4_normal_cg", n5 * (3 * sp + 4 * acc), links);
    pcls[4] = prof_class(pre + ".P_update", n5 * (acc + 2 * sp), 0.0);
    }
    const double l64 = 8.0 * (double)E->vh() * 144.0;
    const std::string rn = "f64.reliable.";
    pcls_rel[0] = prof_class(rn + "K1_minv", n5 * 2 * 192.0, l64);
    pcls_rel[1] = prof_class(rn + "K2_schur_mdinv", n5 * 3 * 192.0, l64);
    pcls_rel[2] = prof_class(rn + "K3_dag_minvdag", n5 * 2 * 192.0, l64);
    pcls_rel[3] = prof_class(rn + "K4_resid", n5 * 4 * 192.0, l64);
    return ODWF_OK;
}

int BatchCG::admit(int slot, const double2* b_ext, double mq_slot, cudaStream_t s, double tol_slot,
                   int max_iter_slot) {
    NvtxRange nv_("odwf.cg.admit");
    idle = false;
    if (slot < 0 || slot >= cap) return fail(ODWF_EINVAL, "admit: bad slot");
    mq[slot] = mq_slot;
    const size_t eb = E->sites5() * 12 * sizeof(double2);
    const double2* bd = b_ext;
    if (!is_device_ptr(b_ext)) {
        // mixed: one copy per slot (read again at every update); FP64: packed at once, one buffer
        int rc = 0;
        bstage = (double2*)E->get_ws("cg.bstage", eb * (mixed ? cap : 1), &rc);
        if (rc) return rc;
        double2* dst = (double2*)((char*)bstage + eb * (mixed ? slot : 0));
        ODWF_CK(cudaMemcpyAsync(dst, b_ext, eb, cudaMemcpyHostToDevice, s));
        bd = dst;
    }
    if (!mixed) {
        ODWF_CK(launch_pack(Sp::F64, bd, B64.ref_sys(slot), E->g, 0, E->ns, 1, s));
        return admit_internal(slot, s, tol_slot, max_iter_slot);
    }
    bsrc[slot] = bd;
    int rc = order_after(s_rel, s);  // the shared FP64 buffers are free
    if (!rc) rc = load_b(slot, s);
    if (!rc) rc = admit_internal(slot, s, tol_slot, max_iter_slot);
    if (!rc) rc = order_after(s, s_rel);  // later updates start after this admission's reads
    return rc;
}

int BatchCG::order_after(cudaStream_t first, cudaStream_t then) {
    ODWF_CK(cudaEventRecord(ev_sync, first));
    ODWF_CK(cudaStreamWaitEvent(then, ev_sync, 0));
    return ODWF_OK;
}

int BatchCG::load_b(int slot, cudaStream_t s) {
    if (mixed && bsrc[slot]) ODWF_CK(launch_pack(Sp::F64, bsrc[slot], B64.ref_sys(0), E->g, 0, E->ns, 1, s));
    return ODWF_OK;
}

int BatchCG::release(int slot) {
    if (slot < 0 || slot >= cap) return fail(ODWF_EINVAL, "release: bad slot");
    active[slot] = 0;
    if (!bsrc.empty()) bsrc[slot] = nullptr;
    st_host[slot].status = kIdle;
    return ODWF_OK;
}

int BatchCG::cancel(int slot, cudaStream_t s) {
    if (slot < 0 || slot >= cap) return fail(ODWF_EINVAL, "cancel: bad slot");
    if (upd[slot]) {
        ODWF_CK(cudaStreamWaitEvent(s, ev_rel[slot], 0));
        upd[slot] = 0;
    }
    ODWF_CK(launch_state(st + slot, 1, 3, 0.0, s));
    return release(slot);
}

int BatchCG::admit_internal(int slot, cudaStream_t s, double tol_slot, int max_iter_slot) {
    idle = false;
    const double tl = tol_slot > 0 ? tol_slot : tol;
    slot_tol[slot] = tl;
    const size_t n5 = E->sites5();
    const int ns = E->ns;
    // per-slot scalars: r = m_q / (2 m0) and a fresh state (written through pinned memory)
    double* rpin = reinterpret_cast<double*>(st_host + 2 * cap) + slot;
    *rpin = mq[slot] / (2.0 * E->m0);
    ODWF_CK(cudaMemcpyAsync(r_dev + slot, rpin, sizeof(double), cudaMemcpyHostToDevice, s));
    SysState init;
    std::memset(&init, 0, sizeof(init));
    init.status = kIdle;
    init.max_iter = max_iter_slot > 0 ? max_iter_slot : max_iter;
    init.delta = delta;
    init.reliable = mixed ? 1 : 0;
    SysState* stage = st_host + cap + slot;  // a slot is re-admitted only after finalize() synchronized
    *stage = init;
    ODWF_CK(cudaMemcpyAsync(st + slot, stage, sizeof(SysState), cudaMemcpyHostToDevice, s));
    // ||b||^2 -> state, then rr = bb, status running
    const FieldRef B = Bref();
    ODWF_CK(launch_vec(Sp::F64, Sp::F64, B, B, n5, ns, 3, 0.0, st, 0, 0, partials, counters, slot, 1, s, nblk));
    ODWF_CK(launch_state(st + slot, 1, 0, tl * tl, s));
    ODWF_CK(launch_vec(Sp::F64, Sp::F64, X64.ref(), X64.ref(), n5, ns, 5, 0.0, st, 0, 0, nullptr, nullptr, slot, 1, s));
    if (!mixed) {
        ODWF_CK(launch_vec(Sp::F64, Sp::F64, B, R64.ref(), n5, ns, 0, 0.0, st, 0, 0, nullptr, nullptr, slot, 1, s));
        ODWF_CK(launch_vec(Sp::F64, Sp::F64, B, P64.ref(), n5, ns, 0, 0.0, st, 0, 0, nullptr, nullptr, slot, 1, s));
    } else {
        ODWF_CK(launch_vec(Sp::F64, Sp::F32, B, Rin.ref(), n5, ns, 6, 0.0, st, 0, 0, nullptr, nullptr, slot, 1, s));
        ODWF_CK(launch_vec(Sp::F32, Sp::F32, Xin.ref(), Xin.ref(), n5, ns, 5, 0.0, st, 0, 0, nullptr, nullptr, slot, 1, s));
        if (v2) {
            ODWF_CK(launch_p_update2(low, ns, Rin.ref(), Pl.ref(), Chil.ref(), E->vh(), 0, E->cf32, r_dev, st, 0, 0,
                                     slot, 1, nullptr, s));
        } else {
            ODWF_CK(launch_vec(Sp::F64, low, B, Pl.ref(), n5, ns, 6, 0.0, st, 0, 0, nullptr, nullptr, slot, 1, s));
        }
    }
    active[slot] = 1;
    n_reliable[slot] = 0;
    st_host[slot].status = kRunning;  // host view until the next poll
    return ODWF_OK;
}

int BatchCG::run_iterations(int k, cudaStream_t s) {
    NvtxRange nv_("odwf.cg.iterations");
    idle = false;
    int lo = cap, hi = -1;
    for (int i = 0; i < cap; ++i)
        if (active[i] && slot_running(i)) {
            lo = std::min(lo, i);
            hi = std::max(hi, i);
        }
    if (hi < 0) return ODWF_OK;
    const int n = hi - lo + 1;
    // direct launches while profiling (per-launch events), on the default streams (not
    // capturable), or when ODWF_GRAPHS=0 is set in the environment
    static const bool graphs_on = [] {
        const char* v = std::getenv("ODWF_GRAPHS");
        return !(v && v[0] == '0');
    }();
    if (!graphs_on || prof_enabled() || s == nullptr || s == cudaStreamLegacy || s == cudaStreamPerThread)
        return launch_iterations(k, lo, n, s);
    const int range[3] = {lo, n, k};
    const std::string key = graph_key + std::string((const char*)range, sizeof(range));
    auto it = H->graphs.find(key);
    if (it == H->graphs.end()) {
        if (H->graphs.size() >= 32) H->drop_graphs();
        const long long c0 = launch_count();
        ODWF_CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
        const int rc = launch_iterations(k, lo, n, s);
        cudaGraph_t g = nullptr;
        const cudaError_t ce = cudaStreamEndCapture(s, &g);
        CgHost::Graph e;
        e.kernels = launch_count() - c0;
        note_launches(-e.kernels);  // captured, not launched
        if (rc || ce != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return rc ? rc : cuda_fail(ce, "cudaStreamEndCapture(CG iterations)");
        }
        const cudaError_t ie = cudaGraphInstantiate(&e.exec, g, 0);
        cudaGraphDestroy(g);
        if (ie != cudaSuccess) return cuda_fail(ie, "cudaGraphInstantiate(CG iterations)");
        it = H->graphs.emplace(key, e).first;
    }
    ODWF_CK(cudaGraphLaunch(it->second.exec, s));
    note_launches(it->second.kernels);
    return ODWF_OK;
}

int BatchCG::launch_iterations(int k, int lo, int n, cudaStream_t s) {
    const size_t n5 = E->sites5();
    for (int it = 0; it < k; ++it) {
        if (!mixed) {
            ODWF_CK(launch_m5_fx(P64.ref(), C64.ref(), E->g, 0, E->ns, r_dev, lo, n, FxOp::B, E->fx_tab, s, st, kRunning));
            const FieldRef f[5] = {C64.ref(), A64.ref(), C64.ref(), A64.ref(), FieldRef{}};
            const Epi e[4] = {Epi::MINV, Epi::SCHUR_NORM_MDINV, Epi::D_MINVDAG, Epi::D_NORMAL_CG};
            for (int h = 0; h < 4; ++h) {
                auto P = params<double>(1 - (h & 1));
                P.gate = 1;
                P.need_status = kRunning;
                P.sys_base = lo;
                P.in = f[h];
                P.out = f[h + 1];
                if (h == 1) P.z = P64.ref();
                if (h == 3) {
                    P.z = C64.ref();
                    P.cg_r = R64.ref();
                    P.cg_x = X64.ref();
                    P.cg_p = P64.ref();
                }
                auto pb_ = prof_begin(pcls[h], s);
                P.prof_count = pb_.dev_count;
                const cudaError_t e_ = launch_hop_fx(P, e[h], n, s);
                prof_end(pb_, s);
                ODWF_CK(e_);
            }
            {
                auto pb_ = prof_begin(pcls[4], s);
                set_vec_prof(pb_.dev_count);
                cudaError_t e_ = launch_vec(Sp::F64, Sp::F64, R64.ref(), P64.ref(), n5, E->ns, 1, 0.0, st, 1, kRunning,
                                            nullptr, nullptr, lo, n, s);
                set_vec_prof(nullptr);
                prof_end(pb_, s);
                ODWF_CK(e_);
            }
        } else if (v2) {
            // With few partials the p update forms beta and the next K1 puts it into the state, which saves
            // a launch; the last iteration of the chunk finalizes before the host looks.
            const int nb = hop_blocks(E->ns, low, 4, E->vh(), n);
            const bool in_update = nb * n <= kBetaInUpdate, last = it + 1 == k;
            int rc = launch_v2_hops(lo, n, s, in_update && it > 0, !in_update || last);
            if (!rc) rc = launch_v2_pupdate(1, lo, n, 1, kRunning, s, in_update && !last ? nb : 0);
            if (rc) return rc;
        } else {
            auto P = params<float>(1);
            P.gate = 1;
            P.need_status = kRunning;
            P.sys_base = lo;
            P.in = Pl.ref();
            P.out = Tl.ref();
            { auto pb_ = prof_begin(pcls[0], s); P.prof_count = pb_.dev_count; ODWF_CK(launch_hop_mixed(P, Epi::MINV, low, lk, n, s)); prof_end(pb_, s); P.prof_count = nullptr; }
            P.p_out = 0;
            P.in = Tl.ref();
            P.z = Pl.ref();
            P.out = Al.ref();
            { auto pb_ = prof_begin(pcls[1], s); P.prof_count = pb_.dev_count; ODWF_CK(launch_hop_mixed(P, Epi::SCHUR_NORM_MDINV, low, lk, n, s)); prof_end(pb_, s); P.prof_count = nullptr; }
            P.p_out = 1;
            P.in = Al.ref();
            P.z = FieldRef{};
            P.out = Cl.ref();
            { auto pb_ = prof_begin(pcls[2], s); P.prof_count = pb_.dev_count; ODWF_CK(launch_hop_mixed(P, Epi::D_MINVDAG, low, lk, n, s)); prof_end(pb_, s); P.prof_count = nullptr; }
            P.p_out = 0;
            P.in = Cl.ref();
            P.z = Al.ref();
            P.out = FieldRef{};
            P.cg_r = Rin.ref();
            P.cg_x = Xin.ref();
            P.cg_p = Pl.ref();
            { auto pb_ = prof_begin(pcls[3], s); P.prof_count = pb_.dev_count; ODWF_CK(launch_hop_mixed(P, Epi::D_NORMAL_CG, low, lk, n, s)); prof_end(pb_, s); P.prof_count = nullptr; }
            {
                auto pb_ = prof_begin(pcls[4], s);
                set_vec_prof(pb_.dev_count);
                cudaError_t e_ = launch_vec(Sp::F32, low, Rin.ref(), Pl.ref(), n5, E->ns, 1, 0.0, st, 1, kRunning,
                                            nullptr, nullptr, lo, n, s);
                set_vec_prof(nullptr);
                prof_end(pb_, s);
                ODWF_CK(e_);
            }
        }
    }
    return ODWF_OK;
}

// One of the hops K1..K4 of a second-generation mixed iteration over slots lo..lo+n-1 (the non-dagger hops
// read chi = B psi).  K3 also forms alpha from K2's partials, K1 beta from nb_prev of K4's.
int BatchCG::launch_v2_hop(int kind, int lo, int n, cudaStream_t s, int nb_prev) {
    auto P = params<float>(1);
    P.gate = 1;
    P.need_status = kRunning;
    P.sys_base = lo;
    const FieldRef ins[4] = {Chil.ref(), Tl.ref(), Al.ref(), Cl.ref()};
    const FieldRef outs[4] = {Tl.ref(), Al.ref(), Cl.ref(), FieldRef{}};
    const FieldRef zs[4] = {FieldRef{}, Pl.ref(), FieldRef{}, Al.ref()};
    const int k = kind - 1;
    P.p_out = (k & 1) ? 0 : 1;
    P.in = ins[k];
    P.out = outs[k];
    P.z = zs[k];
    if (k == 3) {
        P.cg_r = Rin.ref();
        P.cg_x = Xin.ref();
        P.cg_p = Pl.ref();
    }
    P.nb_prev = k == 2 ? hop_blocks(E->ns, low, 2, E->vh(), n) : k == 0 ? nb_prev : 0;
    auto pb_ = prof_begin(pcls[k], s);
    P.prof_count = pb_.dev_count;
    const cudaError_t e_ = launch_hop_prod(P, kind, low, lk, n, s);
    prof_end(pb_, s);
    ODWF_CK(e_);
    return ODWF_OK;
}

// beta of every running system from K4's partials
int BatchCG::launch_v2_beta(int lo, int n, cudaStream_t s) {
    auto pb_ = prof_begin(pcls[5], s);
    const cudaError_t e_ = launch_beta(partials, hop_blocks(E->ns, low, 4, E->vh(), n), nblk, st, kRunning, lo, n, s);
    prof_end(pb_, s);
    ODWF_CK(e_);
    return ODWF_OK;
}

// A kernel of the iteration as the solver replays it, with the sums over partials that it or a launch of its own makes
int BatchCG::launch_v2_kernel(int kind, int lo, int n, cudaStream_t s) {
    const int nb = hop_blocks(E->ns, low, 4, E->vh(), n);
    const bool in_update = nb * n <= kBetaInUpdate;
    if (kind == 5) return launch_v2_pupdate(1, lo, n, 1, kRunning, s, in_update ? nb : 0);
    const int rc = launch_v2_hop(kind, lo, n, s, in_update ? nb : 0);
    return rc || kind != 4 || in_update ? rc : launch_v2_beta(lo, n, s);
}

int BatchCG::launch_v2_hops(int lo, int n, cudaStream_t s, bool prev_beta, bool last_beta) {
    const int nb = prev_beta ? hop_blocks(E->ns, low, 4, E->vh(), n) : 0;
    for (int kind = 1; kind <= 4; ++kind)
        if (const int rc = launch_v2_hop(kind, lo, n, s, nb)) return rc;
    return last_beta ? launch_v2_beta(lo, n, s) : ODWF_OK;
}

// p = r + beta p (mode 1) or p = r (mode 0), chi_p = B p, for the slots whose status is `need`.
int BatchCG::launch_v2_pupdate(int mode, int lo, int n, int gate, int need, cudaStream_t s, int nb) {
    auto pb_ = prof_begin(pcls[4], s);
    const cudaError_t e_ = launch_p_update2(low, E->ns, Rin.ref(), Pl.ref(), Chil.ref(), E->vh(), mode, E->cf32, r_dev,
                                            st, gate, need, lo, n, pb_.dev_count, s, partials, nb, nblk);
    prof_end(pb_, s);
    ODWF_CK(e_);
    return ODWF_OK;
}

int BatchCG::set_state(int slot, const SysState& init, double r, cudaStream_t s) {
    if (slot < 0 || slot >= cap) return fail(ODWF_EINVAL, "set_state: bad slot");
    double* rpin = reinterpret_cast<double*>(st_host + 2 * cap) + slot;
    *rpin = r;
    ODWF_CK(cudaMemcpyAsync(r_dev + slot, rpin, sizeof(double), cudaMemcpyHostToDevice, s));
    SysState* stage = st_host + cap + slot;
    *stage = init;
    ODWF_CK(cudaMemcpyAsync(st + slot, stage, sizeof(SysState), cudaMemcpyHostToDevice, s));
    ODWF_CK(cudaStreamSynchronize(s));
    return ODWF_OK;
}

int BatchCG::poll(cudaStream_t s) {
    ODWF_CK(cudaMemcpyAsync(st_host, st, sizeof(SysState) * cap, cudaMemcpyDeviceToHost, s));
    ODWF_CK(cudaStreamSynchronize(s));
    prof_collect();
    return ODWF_OK;
}

bool BatchCG::slot_running(int i) const {
    const int stt = st_host[i].status;
    return stt == kRunning || stt == kNeedUpdate;
}

bool BatchCG::slot_finished(int i) const {
    const int stt = st_host[i].status;
    return active[i] && (stt == kDone || stt == kBreakdown || stt == kMaxIter);
}

int BatchCG::any_running() const {
    int n = 0;
    for (int i = 0; i < cap; ++i)
        if (active[i] && (slot_running(i) || upd[i])) ++n;
    return n;
}

int BatchCG::resume(cudaStream_t s, bool block) {
    bool any_iterating = false;
    for (int i = 0; i < cap; ++i)
        if (active[i] && !upd[i] && st_host[i].status == kRunning) any_iterating = true;
    for (int i = 0; i < cap; ++i) {
        if (!upd[i]) continue;
        cudaError_t q = cudaEventQuery(ev_rel[i]);
        if (q == cudaErrorNotReady && block && !any_iterating) {
            ODWF_CK(cudaEventSynchronize(ev_rel[i]));  // nothing else to do: wait for this update
            q = cudaSuccess;
        }
        if (q == cudaErrorNotReady) continue;
        if (q != cudaSuccess) return cuda_fail(q, "cudaEventQuery(reliable update)");
        // the iteration stream waits for the update, then the slot rejoins (kRestarting -> kRunning)
        ODWF_CK(cudaStreamWaitEvent(s, ev_rel[i], 0));
        ODWF_CK(launch_state(st + i, 1, 2, 0.0, s));
        upd[i] = 0;
        st_host[i].status = kRunning;  // host view until the next poll
        any_iterating = true;
    }
    return ODWF_OK;
}

// R[slot] = B[slot] - S^dag S X[slot] to FP64 accuracy, |R|^2 -> st[slot].sum (mixed: R and B are the
// shared buffers, B loaded with the slot's right-hand side)
int BatchCG::fp64_residual(int slot, cudaStream_t s) {
    const FieldRef a = mixed ? A1.ref_shared() : A64.ref(), c = mixed ? C1.ref_shared() : C64.ref();
    ODWF_CK(launch_m5_fx(X64.ref(), c, E->g, 0, E->ns, r_dev, slot, 1, FxOp::B, E->fx_tab, s));
    const FieldRef f[5] = {c, a, c, a, Rref()};
    const Epi e[4] = {Epi::MINV, Epi::SCHUR_MDINV, Epi::D_MINVDAG, Epi::D_NORMAL_RESID};
    for (int h = 0; h < 4; ++h) {
        auto P = params<double>(1 - (h & 1));
        P.sys_base = slot;
        P.in = f[h];
        P.out = f[h + 1];
        if (h == 1) P.z = X64.ref();
        if (h == 3) {
            P.z = c;
            P.b = Bref();
        }
        auto pb_ = prof_begin(pcls_rel[h], s);
        P.prof_count = pb_.dev_count;
        const cudaError_t e_ = launch_hop_fx(P, e[h], 1, s);
        prof_end(pb_, s);
        ODWF_CK(e_);
    }
    return ODWF_OK;
}

int BatchCG::service(cudaStream_t s) {
    NvtxRange nv_("odwf.cg.reliable_updates");
    const size_t n5 = E->sites5();
    for (int i = 0; i < cap; ++i) {
        if (!active[i] || upd[i] || st_host[i].status != kNeedUpdate) continue;
        // the update stream starts after this slot's last iteration on s
        ODWF_CK(cudaEventRecord(ev_rel[i], s));
        ODWF_CK(cudaStreamWaitEvent(s_rel, ev_rel[i], 0));
        cudaStream_t r = s_rel;
        if (mixed)  // X64 += rscale x_in, x_in = 0
            ODWF_CK(launch_vec(Sp::F32, Sp::F64, Xin.ref(), X64.ref(), n5, E->ns, 7, 0.0, st, 0, 0, nullptr, nullptr,
                               i, 1, r));
        int rc = load_b(i, r);
        if (!rc) rc = fp64_residual(i, r);
        if (rc) return rc;
        ODWF_CK(launch_state(st + i, 1, 1, tol * tol, r));  // done / max-iter / kRestarting
        if (mixed) {
            ODWF_CK(launch_vec(Sp::F64, Sp::F32, Rref(), Rin.ref(), n5, E->ns, 6, 0.0, st, 1, kRestarting, nullptr,
                               nullptr, i, 1, r));
            if (v2) {
                ODWF_CK(launch_p_update2(low, E->ns, Rin.ref(), Pl.ref(), Chil.ref(), E->vh(), 1, E->cf32, r_dev, st,
                                         1, kRestarting, i, 1, nullptr, r));
            } else {
                ODWF_CK(launch_vec(Sp::F32, low, Rin.ref(), Pl.ref(), n5, E->ns, 1, 0.0, st, 1, kRestarting, nullptr,
                                   nullptr, i, 1, r));
            }
        } else {
            ODWF_CK(launch_vec(Sp::F64, Sp::F64, R64.ref(), P64.ref(), n5, E->ns, 1, 0.0, st, 1, kRestarting, nullptr,
                               nullptr, i, 1, r));
        }
        ODWF_CK(cudaEventRecord(ev_rel[i], r));
        upd[i] = 1;
        n_reliable[i] += 1;
        st_host[i].status = kRestarting;  // host view until the next poll
    }
    return ODWF_OK;
}

int BatchCG::finalize(int slot, double2* x_ext, cudaStream_t s, double* true_resid) {
    NvtxRange nv_("odwf.cg.finalize");
    if (upd[slot]) {
        ODWF_CK(cudaStreamWaitEvent(s, ev_rel[slot], 0));
        upd[slot] = 0;
    }
    ODWF_CK(cudaMemcpyAsync(st_host + slot, st + slot, sizeof(SysState), cudaMemcpyDeviceToHost, s));
    ODWF_CK(cudaStreamSynchronize(s));
    const int stt = st_host[slot].status;
    if (stt != kDone && stt != kMaxIter) {
        // breakdown (or an unfinished slot): fold and recompute the true residual
        int rc = ODWF_OK;
        if (mixed) {
            ODWF_CK(launch_vec(Sp::F32, Sp::F64, Xin.ref(), X64.ref(), E->sites5(), E->ns, 7, 0.0, st, 0, 0, nullptr,
                               nullptr, slot, 1, s));
            rc = order_after(s_rel, s);  // the shared FP64 buffers are free
            if (!rc) rc = load_b(slot, s);
        }
        if (!rc) rc = fp64_residual(slot, s);
        if (!rc && mixed) rc = order_after(s, s_rel);
        if (rc) return rc;
    }
    if (x_ext) ODWF_CK(launch_unpack(Sp::F64, X64.ref_sys(slot), x_ext, E->g, 0, E->ns, 1, s));
    ODWF_CK(cudaMemcpyAsync(st_host + slot, st + slot, sizeof(SysState), cudaMemcpyDeviceToHost, s));
    ODWF_CK(cudaStreamSynchronize(s));
    idle = true;
    const SysState& S = st_host[slot];
    if (true_resid) *true_resid = S.bb > 0 ? std::sqrt(S.sum / S.bb) : 0.0;
    return ODWF_OK;
}

}  // namespace odwf
