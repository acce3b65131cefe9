"""The performance cases of the framework: what a search does with it, through its public entry points.

A search whitens every block of strain, filters it through a reduced basis, screens (template, bin)
pairs and reconstructs the survivors (one block, sub-banks, or a recorded batch), compares with the
template method, and refines what it found. Inputs stand for that use: TaylorF2 banks, coloured
Gaussian noise with a chirp in it, a basis orthonormalised from templates of the bank. They are made
with torch from the seed alone; lists that the library returns in no set order are put in order
(template, then time) on the device or, for host buffers, on the host.
"""
import math

import numpy as np
import torch

from paper_2110_13115_gb300 import api, inputs

FS, F_LOW = 2048.0, 30.0
SNR = 10.0  # of the one chirp in an ordinary block, the lightest of the bank: most of what is filtered is noise
PRECISIONS = ["fp16_split_a", "fp16_split", "fp16", "bf16_split", "bf16", "fp32"]


def listed():
    return [
        # one 256-s block's data FFT and whitening: the smallest call, launches and the read-back
        dict(name="whiten", kind="whiten", n=1 << 19),
        # a low-latency search: one 16-s block, a small bank, the whole filter in one call
        dict(name="filter-small", kind="filter", n=1 << 14, T=64, k=40, w=8, precision="fp16_split", rho_i=4.0,
             rho_ii=5.5),
        # basis series of a 64-s block in a batch of segments (ragged k, wide bins)
        dict(name="basis-64s", kind="basis", n=1 << 17, k=77, w=16),
        # basis series of a 256-s block for one sub-bank of the 10,000-template bank
        dict(name="basis-256s", kind="basis", n=1 << 19, k=201, w=8),
        # the screening product of the whole bank on one basis
        dict(name="stage1-bank", kind="stage1", n=1 << 19, T=10000, k=256, w=8, precision="fp16_split_a", rho_i=4.8),
        # reconstruction of a sub-bank's candidates in a block with loud signals, the benchmark's screening threshold
        dict(name="stage2-subbank", kind="stage2", n=1 << 19, T=2500, k=201, w=8, rho_i=4.373, rho_ii=15.0, chirps=6,
             snr=20.0),
        # the template method, which a search keeps as its comparator and for follow-up
        dict(name="template-method", kind="plain", n=1 << 19, T=200, w=8, rho_ii=6.0),
        # the first stage by the template method
        dict(name="folded", kind="folded", n=1 << 18, T=400, w=8, rho_i=5.5),
        # |SNR|^2 of candidates and its gradient through autograd (a sampler or an optimiser of the user's own)
        dict(name="gradient", kind="gradient", n=1 << 19, T=500),
        # the built-in ascent on the candidates of a 64-s block
        dict(name="refine", kind="refine", n=1 << 17, T=512, steps=20),
        # a recorded batch: blocks of three lengths replayed as one graph
        dict(name="batch", kind="batch", n=1 << 18, T=3000, k=128, w=8, precision="fp16_split_a", rho_i=4.373,
             rho_ii=6.0, blocks=9),
        # the benchmark's block: 10,000 templates in four sub-banks, host strain in, host triggers out
        dict(name="banks-256s", kind="banks", n=1 << 19, T=10000, k=563, w=8, precision="fp16_split_a", rho_i=4.373,
             rho_ii=6.0),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the ranges above: block lengths 2^12..2^19 (whitening to 2^20), ragged T and k."""
    kind = rng.choice(["whiten", "filter", "basis", "basis", "stage1", "stage2", "plain", "folded", "gradient", "refine",
                       "batch", "banks"])
    n = 1 << rng.randint(13, 19)
    w = rng.choice([1, 2, 4, 8, 8, 16])
    k, T = _log(rng, 16, 256), _log(rng, 64, 2500)
    prec = rng.choice(PRECISIONS[:2] + PRECISIONS)
    rho_i = round(rng.uniform(5.0, 5.5), 3)
    if kind == "whiten":
        return dict(kind=kind, n=1 << rng.randint(12, 20))
    if kind == "basis":
        return dict(kind=kind, n=n, k=k, w=w)
    if kind == "stage1":
        return dict(kind=kind, n=n, T=max(T, k), k=k, w=w, precision=prec, rho_i=rho_i)
    if kind == "stage2":
        snr = round(rng.uniform(8, 20), 1)
        return dict(kind=kind, n=n, T=max(T, k), k=k, w=w, rho_i=round(rho_i - 0.6, 3), rho_ii=0.75 * snr,
                    chirps=rng.randint(1, 6), snr=snr)
    if kind == "plain":
        return dict(kind=kind, n=n, T=_log(rng, 16, 200), w=w, rho_ii=6.0)
    if kind == "folded":
        return dict(kind=kind, n=max(n, 1 << 14), T=_log(rng, 16, 400), w=rng.choice([2, 4, 8, 16]), rho_i=rho_i)
    if kind == "gradient":
        return dict(kind=kind, n=n, T=_log(rng, 8, 500))
    if kind == "refine":
        return dict(kind=kind, n=1 << rng.randint(13, 17), T=_log(rng, 16, 500), steps=rng.randint(5, 20))
    if kind == "batch":
        return dict(kind=kind, n=1 << rng.randint(15, 18), T=max(T, k), k=k, w=w, precision=prec, rho_i=rho_i,
                    rho_ii=6.0, blocks=rng.randint(3, 9))
    if kind == "banks":
        k = rng.randint(64, 400)
        return dict(kind=kind, n=1 << rng.randint(16, 19), T=max(_log(rng, 400, 6000), 8 * k), k=k, w=rng.choice([4, 8, 16]),
                    precision=rng.choice(PRECISIONS[:2]), rho_i=rho_i, rho_ii=6.0)
    return dict(kind=kind, n=min(n, 1 << 18), T=max(T, k), k=k, w=w, precision=prec, rho_i=rho_i, rho_ii=6.0)


# --- inputs ------------------------------------------------------------------------------------

def _grid(n):
    return inputs.Grid(FS, n, F_LOW)


def _psd(n):
    return torch.from_numpy(inputs.analytic_psd(_grid(n))).cuda()


def _masses(n, T, seed):
    """Bank parameters [T, 4]; short blocks take the heavier banks whose templates fit into them."""
    lo = 3.0 if n >= 1 << 18 else 5.0 if n >= 1 << 17 else 8.0 if n >= 1 << 16 else 10.0
    p = inputs.draw_bank(inputs.BankSpec(T, lo, 50.0 if n >= 1 << 16 else 30.0, 0.5, 3), seed=seed)
    mt = p.sum(axis=1) - p[:, 2] - p[:, 3]
    tau = (p[:, 0] * p[:, 1] / mt ** 2) ** -1 * mt ** (-5.0 / 3.0)  # ascending Newtonian chirp time
    return p[np.argsort(tau, kind="stable")]


def _phase(f, p):
    """Psi(f) of rows p = (m1, m2, chi1, chi2) through 1.5PN, without coalescence time and phase; float64 [T, len(f)]."""
    m1, m2, x1, x2 = (p[:, i] for i in range(4))
    mt = m1 + m2
    eta, q1, q2 = m1 * m2 / mt ** 2, m1 / mt, m2 / mt
    u = math.pi * mt * inputs.MSUN_S  # v^3 = u f
    so = (x1 * (113 * q1 * q1 + 75 * eta) + x2 * (113 * q2 * q2 + 75 * eta)) / 12
    c0, c2, c3 = 3 / (128 * eta), (20 / 9) * (743 / 336 + 11 * eta / 4), 4 * so - 16 * math.pi
    rows = torch.stack([c0 * u ** (-5 / 3), c0 * c2 / u, c0 * c3 * u ** (-2 / 3), torch.full_like(u, -math.pi / 4)], 1)
    return rows @ torch.stack([f ** (-5 / 3), 1 / f, f ** (-2 / 3), torch.ones_like(f)])


def _rows(n, params, psd, dtype=torch.complex64):
    """Whitened unit-norm templates [T, n/2]."""
    df, half = FS / n, n // 2
    j0 = int(math.ceil(F_LOW / df))
    j1 = min(half, int(1 / (6 ** 1.5 * math.pi * float(params[:, :2].sum(axis=1).min()) * inputs.MSUN_S) / df) + 2)
    f = torch.arange(j0, j1, device="cuda", dtype=torch.float64) * df
    amp = f ** (-7 / 6) * torch.sqrt(4 * df / psd[j0:j1])
    out = torch.zeros((len(params), half), dtype=dtype, device="cuda")
    step = max(1, (1 << 26) // (j1 - j0))
    for t in range(0, len(params), step):
        p = torch.from_numpy(params[t:t + step]).cuda()
        cut = 1 / (6 ** 1.5 * math.pi * (p[:, :1] + p[:, 1:2]) * inputs.MSUN_S)
        a = amp[None] * (f[None] < cut)
        a = a / torch.linalg.vector_norm(a, dim=1, keepdim=True)
        out[t:t + step, j0:j1] = torch.polar(a, -_phase(f, p)).to(dtype)
    return out


def _strain(n, seed, params, snr, chirps=1):
    """Coloured Gaussian noise and chirps of the given optimal SNR, spread over the valid half; float32 [n], and the PSD."""
    g = torch.Generator("cuda").manual_seed(seed)
    psd, half = _psd(n), n // 2
    x = torch.randn((2, half), generator=g, device="cuda", dtype=torch.float64)
    df = FS / n
    f = torch.arange(half, device="cuda", dtype=torch.float64) * df
    amp = torch.where(f >= F_LOW / 2, torch.sqrt(psd[:half] * n / FS / 4), torch.zeros_like(f))
    amp[0] = 0
    s = amp * torch.complex(x[0], x[1])
    if snr:
        h = _rows(n, params[None], psd, torch.complex128)[0] / torch.sqrt(4 * df / psd[:half])
        h = torch.where(torch.isfinite(h.real), h, torch.zeros_like(h))
        for c in range(chirps):
            tc = (0.5 + 0.5 * (c + 0.5) / chirps) * n / FS
            s = s + snr * h * torch.polar(torch.ones_like(f), -2 * math.pi * f * tc)
    s = torch.cat([s, s.new_zeros(1)])
    return (torch.fft.irfft(s, n=n) * FS).float(), psd


def _white64(n, strain, psd):
    """s_hat in 64 bits: sqrt(4 df / S_j) dt DFT(strain)[j] on 0 < j < n/2."""
    s = torch.fft.rfft(strain.double())[:n // 2] / FS * torch.sqrt(4 * FS / n / psd[:n // 2])
    s[0] = 0
    return s


def _basis(n, params, psd, k, rows=None):
    """k basis vectors orthonormalised from templates spread over the bank, and the bank's coefficients on them."""
    rows = _rows(n, params, psd) if rows is None else rows
    piv = rows[torch.linspace(0, len(params) - 1, k, device="cuda").long()]
    gram = (piv @ piv.mH).to(torch.complex128) + 1e-3 * torch.eye(k, device="cuda")
    inv = torch.linalg.inv(torch.linalg.cholesky(gram)).to(torch.complex64)
    vec = (inv @ piv).contiguous()
    return api.Basis(vec, (rows @ vec.mH).contiguous(), n)


def _series(s_hat, rows):
    """sum_j s_hat[j] conj(row[j]) exp(2 pi i j m / n) on the valid half; in the precision of its inputs."""
    n = 2 * s_hat.numel()
    out = torch.empty((len(rows), n // 2), dtype=s_hat.dtype, device="cuda")
    step = max(1, (1 << 25) // n)
    for t in range(0, len(rows), step):
        out[t:t + step] = (torch.fft.ifft(s_hat * rows[t:t + step].to(s_hat.dtype).conj(), n=n) * n)[:, n // 2:]
    return out


def _candidates(coeff, bavg, rho_i, nb):
    """Candidates in the order in which a tiled first stage finds them (blocks of bins, then of templates)."""
    T = len(coeff)
    mask = torch.zeros(((T + 63) // 64 * 64, (nb + 255) // 256 * 256), dtype=torch.bool, device="cuda")
    for t in range(0, T, 512):
        mask[t:t + 512, :nb][:min(512, T - t)] = (coeff[t:t + 512].conj() @ bavg).abs() >= rho_i
    m = mask.view(-1, 4, 16, mask.shape[1] // 256, 8, 32).permute(3, 0, 1, 4, 2, 5)
    i = m.nonzero()
    tm, b = i[:, 1] * 64 + i[:, 2] * 16 + i[:, 4], i[:, 0] * 256 + i[:, 3] * 32 + i[:, 5]
    rec = torch.zeros((len(i), 4), dtype=torch.int32, device="cuda")
    rec[:, 0], rec[:, 1] = tm.int(), (nb + b).int()
    return rec


def _refine_setup(case, seed):
    n, T = case["n"], case["T"]
    rng = np.random.default_rng(seed)
    src = np.array([rng.uniform(12, 25), rng.uniform(8, 12), 0.0, 0.0])
    strain, psd = _strain(n, seed, src, 14.0)
    eta = src[0] * src[1] / (src[0] + src[1]) ** 2
    mc = (src[0] + src[1]) * eta ** 0.6
    th = np.column_stack([mc * (1 + 2e-3 * rng.standard_normal(T)), np.clip(eta * (1 + 0.02 * rng.standard_normal(T)), 0.1, 0.2499),
                          0.75 * n / FS + 2e-3 * rng.standard_normal(T), rng.uniform(0, 2 * np.pi, T)])
    return _white64(n, strain, psd).to(torch.complex64), psd, torch.from_numpy(th).cuda()


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "whiten":
        strain, psd = _strain(n, seed, None, 0.0)
        d = api.make_desc(FS, n, 1, 1, w=1)
        return dict(case, d=d, strain=strain, psd=psd, ws=api.workspace(d))
    if kind in ("gradient", "refine"):
        s_hat, psd, th = _refine_setup(case, seed)
        rd = api.make_refine_desc(FS, n, F_LOW, pn_order=2, steps=case.get("steps", 0))
        return dict(case, d=rd, s_hat=s_hat, psd=psd, theta=th)
    w = case["w"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    if kind == "banks":
        return _prepare_banks(case, seed)
    if kind == "basis":
        params = _masses(n, 4 * case["k"], seed)
        strain, psd = _strain(n, seed, params[-1], SNR)
        basis = _basis(n, params, psd, case["k"])
        d = api.make_desc(FS, n, case["k"], len(params), w=w)
        return dict(case, d=d, basis=basis, s_hat=_white64(n, strain, psd).to(torch.complex64), ws=api.workspace(d))
    params = _masses(n, case["T"], seed)
    strain, psd = _strain(n, seed, params[len(params) // 2 if "chirps" in case else -1], case.get("snr", SNR),
                          case.get("chirps", 1))
    if kind in ("plain", "folded"):
        d = api.make_desc(FS, n, 1, case["T"], w=w, rho_i=case.get("rho_i", 0.0), rho_ii=case.get("rho_ii", 0.0),
                          cand_capacity=1 << 22)
        st = dict(case, d=d, rows=_rows(n, params, psd), strain=strain, psd=psd)
        if kind == "plain":
            st["ws"], st["out"] = api.workspace(d), torch.empty(24 << 20, dtype=torch.uint8, device="cuda")
        else:
            st["ws"] = torch.empty(api.rb_folded_plan(d), dtype=torch.uint8, device="cuda")
            st["out"] = torch.empty(16 << 22, dtype=torch.uint8, device="cuda")
        return st
    basis = _basis(n, params, psd, case["k"])
    d = api.make_desc(FS, n, case["k"], case["T"], w=w, precision=case.get("precision", "fp16_split_a"),
                      rho_i=case["rho_i"], rho_ii=case.get("rho_ii", 5.0), cand_capacity=1 << 22)
    api.rb_pack_coeff(d, basis)
    st = dict(case, d=d, basis=basis, psd=psd, ws=api.workspace(d, host=kind == "filter"))
    if kind == "filter":
        return dict(st, host=strain.cpu().pin_memory(), out=_host_list())
    beta = _series(_white64(n, strain, psd).to(torch.complex64), basis.vectors)
    bavg = beta.view(case["k"], -1, w).mean(2).contiguous()
    if kind == "stage1":
        st["bavg"] = bavg
    else:
        st["beta"], st["cand"] = beta, _candidates(basis.coeff, bavg, case["rho_i"], n // (2 * w))
    return st


def _prepare_batch(case, seed):
    """Blocks of n, n/2 and n/4 samples, a basis per length over one bank."""
    params = _masses(case["n"] // 4, case["T"], seed)
    descs, bases, blocks, psds = [], [], [], []
    for i in range(3):
        n = case["n"] >> i
        psds.append(_psd(n))
        basis = _basis(n, params, psds[-1], case["k"])
        d = api.make_desc(FS, n, case["k"], case["T"], w=case["w"], precision=case["precision"], rho_i=case["rho_i"],
                          rho_ii=case["rho_ii"], cand_capacity=1 << 21)
        api.rb_pack_coeff(d, basis)
        descs.append(d)
        bases.append(basis)
    for b in range(case["blocks"]):
        i, n = b % 3, case["n"] >> (b % 3)
        x, _ = _strain(n, seed + 7919 * (b + 1), params[-1], SNR if b == 1 else 0.0)
        blocks.append(api.Block(x, psds[i], i, sample_offset=b * case["n"], block_id=b))
    return dict(case, handle=api.Batch(descs, bases, blocks, capacity=1 << 20), blocks=blocks, bases=bases)


def _prepare_banks(case, seed):
    """Four sub-banks in order of chirp time; the basis vectors shared out as the benchmark's (the middle parts need fewer)."""
    n, w = case["n"], case["w"]
    params = _masses(n, case["T"], seed)
    strain, psd = _strain(n, seed, params[-1], SNR)
    ks = [max(8, int(case["k"] * s / 563)) for s in (201, 106, 85, 171)]
    descs, bases, off = [], [], [case["T"] * i // 4 for i in range(5)]
    for i in range(4):
        p = params[off[i]:off[i + 1]]
        basis = _basis(n, p, psd, ks[i])
        d = api.make_desc(FS, n, ks[i], len(p), w=w, precision=case["precision"], rho_i=case["rho_i"], rho_ii=case["rho_ii"],
                          cand_capacity=1 << 21)
        api.rb_pack_coeff(d, basis)
        descs.append(d)
        bases.append(basis)
    return dict(case, descs=descs, bases=bases, psd=psd, host=strain.cpu().pin_memory(),
                out=_host_list(), ws=api.banks_workspace(descs, host=True))


def _host_list(room=1 << 20):
    """A pinned host buffer for triggers, as records."""
    return torch.empty(24 * room, dtype=torch.uint8).pin_memory().numpy().view(api.TRIGGER_NP)


# --- one pass -------------------------------------------------------------------------------------

ROOM = 1 << 18  # records of a returned list; what it does not fill is zero


def _ordered(rec, key):
    out = torch.zeros((ROOM, rec.shape[1]), dtype=torch.int64, device="cuda")
    order = torch.sort(key)[1][:ROOM]
    torch.index_select(rec, 0, order, out=out[:len(order)])
    return out, out.view(torch.float32)


def _triggers(buf, n):
    """Trigger records in order of (block, template, sample): sample, template and block, (SNR, phase)."""
    rec = buf.view(torch.int64).view(-1, 3)[:n]
    sample, tmpl, _ = rec.unbind(1)
    out, real = _ordered(rec, torch.add(sample, tmpl, alpha=1 << 24))
    return out[:, 0], out[:, 1], real[:, 4:]


def _host_triggers(rec, n):
    """The same of a host list."""
    out = np.zeros(ROOM, dtype=api.TRIGGER_NP)
    rec = rec[:n]
    out[:n] = rec[np.argsort((rec["tmpl"].astype(np.int64) << 24) + rec["sample"])][:ROOM]
    return out["sample"], out["tmpl"], out["snr"], out["phase"]


def _cands(buf, n):
    """Candidate records in order of (bin, template): template and bin, SNR."""
    rec = buf.view(torch.int64).view(-1, 2)[:n]
    out, real = _ordered(rec, rec[:, 0])
    return out[:, 0], real[:, 2]


def run(s):
    kind = s["kind"]
    if kind == "whiten":
        return api.rb_whiten(s["d"], s["strain"], s["psd"], ws=s["ws"])
    if kind == "basis":
        return api.rb_basis_filter(s["d"], s["basis"], s["s_hat"], ws=s["ws"])
    if kind == "stage1":
        return _cands(*api.rb_stage1(s["d"], s["basis"], s["bavg"], ws=s["ws"]))
    if kind == "stage2":
        return _triggers(*api.rb_stage2(s["d"], s["basis"], s["beta"], s["cand"], len(s["cand"]), ws=s["ws"], capacity=1 << 22))
    if kind == "filter":
        return _host_triggers(s["out"], api.rb_filter_host(s["d"], s["basis"], s["host"], s["psd"], s["out"], ws=s["ws"]))
    if kind == "plain":
        return _triggers(*api.rb_filter_plain(s["d"], s["rows"], s["strain"], s["psd"], capacity=1 << 20, ws=s["ws"], trig=s["out"]))
    if kind == "folded":
        return _cands(*api.rb_stage1_folded(s["d"], s["rows"], s["strain"], s["psd"], ws=s["ws"], cand=s["out"]))
    if kind == "gradient":
        th = s["theta"].detach().requires_grad_(True)
        J = api.peak_snr2(th, s["s_hat"], s["psd"], s["d"])
        J.sum().backward()
        return J.detach(), th.grad
    if kind == "refine":
        return api.rb_refine(s["d"], s["s_hat"], s["psd"], s["theta"])
    if kind == "batch":
        return _triggers(*s["handle"].run())
    return _host_triggers(*api.rb_filter_banks(s["descs"], s["bases"], s["host"], s["psd"], capacity=1 << 20, ws=s["ws"],
                                               trig=s["out"], host=True))


# --- the same in 64 bits --------------------------------------------------------------------------

def _exact_triggers(series_of, hits, w, thr, offset=0, block=0):
    """Triggers of the windows hits = (tmpl, bin) from series_of(tmpl, bin) -> complex128 [len, w]."""
    t, b, z = [], [], []
    for i in range(0, max(1, len(hits)), 1 << 15):
        h = hits[i:i + (1 << 15)]
        v = series_of(h[:, 0], h[:, 1])
        m = v.abs().argmax(1)
        best = v.gather(1, m[:, None])[:, 0]
        keep = best.abs() >= thr
        t.append(h[keep, 0])
        b.append(h[keep, 1] * w + m[keep])
        z.append(best[keep])
    t, m, z = torch.cat(t), torch.cat(b) + offset, torch.cat(z)
    tm = t + (block << 32)
    o = torch.argsort(tm * (1 << 24) + m)
    return torch.stack([z.abs(), z.angle()], 1)[o]


def _list(values):
    """As _ordered: the values with zeros behind them."""
    out = torch.zeros((ROOM, *values.shape[1:]), dtype=torch.float64, device="cuda")
    out[:min(ROOM, len(values))] = values[:ROOM]
    return out


def _reconstruct(coeff, beta, w, n):
    """series_of for the second stage: conj(a_t) . beta over a bin's samples, in 64 bits."""
    b = beta.view(len(beta), -1, w)
    first = n // (2 * w)

    def of(t, i):
        out = []
        for c in range(0, len(t), 2048):
            out.append(torch.einsum("ck,kcw->cw", coeff[t[c:c + 2048]].conj().to(torch.complex128), b[:, i[c:c + 2048] - first].to(torch.complex128)))
        return torch.cat(out) if out else torch.zeros((0, w), dtype=torch.complex128, device="cuda")
    return of


def _exact_block(strain, psd, basis, case, offset=0, block=0):
    """The hierarchical filter of one block in 64 bits."""
    n, w = basis.n, case["w"]
    beta = _series(_white64(n, strain, psd), basis.vectors)
    bavg = beta.view(len(beta), -1, w).mean(2)
    hits = []
    for t in range(0, basis.n_templates, 256):
        h = ((basis.coeff[t:t + 256].to(torch.complex128).conj() @ bavg).abs() >= case["rho_i"]).nonzero()
        hits.append(h + torch.tensor([t, n // (2 * w)], device="cuda"))
    return _exact_triggers(_reconstruct(basis.coeff, beta, w, n), torch.cat(hits), w, case["rho_ii"], offset, block)


def _objective(theta, cut, j0, s_hat, psd, n):
    """J and its gradient at theta [T, 4], support below cut [T]; 64 bits."""
    df = FS / n
    j1 = min(n // 2, int(float(cut.max()) / df) + 2)
    f = torch.arange(j0, j1, device="cuda", dtype=torch.float64)[None] * df
    amp = f ** (-7 / 6) * torch.sqrt(4 * df / psd[None, j0:j1])
    J, G = [], []
    for i in range(0, len(theta), 64):
        mc, eta, tc, ph = (theta[i:i + 64, c:c + 1] for c in range(4))
        mt = mc * eta ** -0.6 * inputs.MSUN_S
        v = (math.pi * mt * f) ** (1 / 3)
        c2 = (20 / 9) * (743 / 336 + 11 * eta / 4)
        pn = 3 / (128 * eta) * (v ** -5 + c2 * v ** -3)
        a = amp * (f < cut[i:i + 64, None])
        term = s_hat[None, j0:j1].to(torch.complex128) * torch.polar(a, 2 * math.pi * f * tc - ph - math.pi / 4 + pn)
        dm = (-5 * v ** -5 - 3 * c2 * v ** -3) / (128 * eta * mt)
        de = -pn / eta + 3 / (128 * eta) * (55 / 9) * v ** -3
        d = [dm * mt / mc, de - 0.6 * dm * mt / eta, 2 * math.pi * f.expand_as(v), -torch.ones_like(v)]
        z, s2 = term.sum(1), (a * a).sum(1)
        J.append(z.abs() ** 2 / s2)
        G.append(torch.stack([2 * (z.conj() * (1j * x * term).sum(1)).real / s2 for x in d], 1))
    return torch.cat(J), torch.cat(G)


def _cutoff(theta):
    return 1 / (6 ** 1.5 * math.pi * theta[:, 0] * theta[:, 1] ** -0.6 * inputs.MSUN_S)


def _ascend(theta, s_hat, psd, n, steps):
    """The documented ascent: normalised gradient in scaled coordinates, a step kept only if J grows."""
    cut, j0 = _cutoff(theta), int(math.ceil(F_LOW * n / FS))
    scale = torch.stack([theta[:, 0], *(torch.full_like(theta[:, 0], x) for x in (1.0, 0.01, 1.0))], 1)
    u, alpha = theta / scale, torch.full_like(theta[:, 0], 1e-3)
    J, g = _objective(theta, cut, j0, s_hat, psd, n)
    for _ in range(steps):
        gu = g * scale
        t = u + alpha[:, None] * gu / torch.linalg.vector_norm(gu, dim=1, keepdim=True)
        t[:, 1].clamp_(0.05, 0.25)
        Jt, gt = _objective(t * scale, cut, j0, s_hat, psd, n)
        up = Jt > J
        u, g, J = torch.where(up[:, None], t, u), torch.where(up[:, None], gt, g), torch.where(up, Jt, J)
        alpha = torch.where(up, torch.clamp(2 * alpha, max=0.05), alpha / 2)
    return u * scale, J


def exact(case, seed):
    """run()'s floating outputs in 64 bits (whole numbers are compared as they are)."""
    s = prepare(case, seed)
    kind, n = case["kind"], case["n"]
    if kind == "whiten":
        return _white64(n, s["strain"], s["psd"])
    if kind == "basis":
        beta = _series(s["s_hat"].to(torch.complex128), s["basis"].vectors)
        return beta, beta.view(len(beta), -1, case["w"]).mean(2)
    if kind == "stage1":
        return None  # the list depends on the screening precision that the caller chose
    if kind == "stage2":
        c = s["cand"].long()
        return None, None, _list(_exact_triggers(_reconstruct(s["basis"].coeff, s["beta"], case["w"], n), c[:, :2], case["w"],
                                                 case["rho_ii"]))
    if kind == "filter":
        z = _list(_exact_block(s["host"].cuda(), s["psd"], s["basis"], case))
        return None, None, z[:, 0], z[:, 1]
    if kind in ("plain", "folded"):
        z = _series(_white64(n, s["strain"], s["psd"]), s["rows"]).view(case["T"], -1, case["w"])
        if kind == "folded":
            r = z.mean(2).abs().T
            return None, _list(r[r >= case["rho_i"]])
        hits = (z.abs().amax(2) >= case["rho_ii"]).nonzero()
        return None, None, _list(_exact_triggers(lambda t, b: z[t, b], hits, case["w"], case["rho_ii"], n // 2))
    if kind == "gradient":
        return _objective(s["theta"], _cutoff(s["theta"]), int(math.ceil(F_LOW * n / FS)), s["s_hat"], s["psd"], n)
    if kind == "refine":
        return _ascend(s["theta"], s["s_hat"], s["psd"], n, case["steps"])
    if kind == "batch":
        return None, None, _list(torch.cat([_exact_block(b.strain, b.psd, s["bases"][b.basis], case, b.sample_offset, b.block_id)
                                            for b in s["blocks"]]))
    z = _list(torch.cat([_exact_block(s["host"].cuda(), s["psd"], b, case) for b in s["bases"]]))
    return None, None, z[:, 0], z[:, 1]


def work(case):
    """Bytes and operations of one pass: inputs and outputs once; n log2 n transforms of one-sided data."""
    kind, n = case["kind"], case["n"]
    half, lg, T, w, k = n // 2, math.log2(n), case.get("T", 1), case.get("w", 1), case.get("k", 1)
    nb = half // w
    whiten = (4 * n + 8 * half + 8 * half, 2.5 * n * lg)
    basis = (k * (16 * half + 8 * nb) + 8 * half, k * (6 * half + 2.5 * n * lg))
    stage1 = (8 * T * k + 8 * k * nb, 8.0 * T * k * nb)
    if kind == "whiten":
        b, f = whiten
    elif kind == "basis":
        b, f = basis
    elif kind == "stage1":
        b, f = stage1
    elif kind == "stage2":  # candidates: about one bin in a hundred
        c = 0.01 * T * nb
        b, f = 16 * c + 8 * T * k + 8 * k * half, 8.0 * c * w * k
    elif kind in ("plain", "folded"):
        b = whiten[0] + 8 * T * half
        f = whiten[1] + T * (6 * half + (2.5 * n * lg if kind == "plain" else 5 * n / w * math.log2(n / w)))
    elif kind in ("gradient", "refine"):  # points from f_low to about 200 Hz; phase, sine and cosine, five sums
        pts = min(half, 170.0 * n / FS)
        b, f = 16 * half + 64 * T, 60.0 * pts * T * (2 if kind == "gradient" else 1 + case["steps"])
    elif kind == "batch":
        b = f = 0
        for i in range(case["blocks"]):
            h = half >> (i % 3)
            b += 4 * 2 * h + 8 * h + 8 * T * k + k * 8 * h
            f += k * 5 * h * math.log2(2 * h) + 8.0 * T * k * h / w
    elif kind == "banks":  # each sub-bank a quarter of the templates with its own vectors
        b, f = 4 * n + 8 * half + 8 * k * half + 2 * T * k, k * (6 * half + 2.5 * n * lg) + 2.0 * T * k * nb
    else:
        b, f = 4 * n + 8 * half + 8 * k * half + 8 * T * k, basis[1] + stage1[1]
    return {"bytes": float(b), "flops": float(f)}
