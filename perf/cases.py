"""The work that users of this library have it do, as cases that can be timed.

Four kinds of call, each through the package's public entry points:

``step``       the batched cluster update, the method's hot path: a state is
               put in place (``load_device``), all clusters of one iteration
               are updated (``step``), and the result is read back
               (``mps_to_host``).  The sites of an updated cluster are only
               defined up to a unitary on each inner bond, so the updated
               state is returned as the clusters' theta tensors,
               diag(lambda_L) B_q ... B_{q+k-1}, next to the fidelities, the
               spectra of the new bonds and the bond dimensions.
``circuit``    a whole simulation from |0...0> (``simulate``) and amplitudes
               of its final state.
``amplitude``  amplitudes of a stored state, as sampling and checks ask for.
``split2``     the two-site split that allocates nothing (``split2_noalloc``).

Sizes are those of the repository's own configurations and tests: chi_max from
a few to 1024, clusters of 2 to 4 sites (up to 8 in whole runs), cutoffs 0 to
1e-12, both precisions.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2502_19289_gb300 as P

H, S, T, X14, CNOT, CZ = 1, 5, 6, 8, 10, 12


def listed():
    return [
        # the smallest iteration: early layers, or a few clusters of a short chain
        dict(name="step_chi8_k2", kind="step", chi=8, k=2, clusters=3, precision="fp32",
             spectrum="decaying", decades=6.0, cutoff=1e-8, ragged=False),
        # many narrow clusters of several sites: packed circuits, sparse layers
        dict(name="step_chi24_k4_ragged", kind="step", chi=24, k=4, clusters=16, precision="fp32",
             spectrum="decaying", decades=8.0, cutoff=1e-8, ragged=True),
        # complex128 mode, for the small and medium widths it is meant for
        dict(name="step_chi64_k3_fp64", kind="step", chi=64, k=3, clusters=4, precision="fp64",
             spectrum="decaying", decades=8.0, cutoff=1e-10, ragged=False),
        # medium bonds that are no multiple of anything
        dict(name="step_chi100_k3_ragged", kind="step", chi=100, k=3, clusters=8, precision="fp32",
             spectrum="decaying", decades=8.0, cutoff=1e-8, ragged=True),
        # the chi_max = 256 configuration near saturation
        dict(name="step_chi256_k3", kind="step", chi=256, k=3, clusters=6, precision="fp32",
             spectrum="decaying", decades=8.0, cutoff=1e-10, ragged=False),
        # the chi_max = 512 configuration, two-site clusters of a dense layer
        dict(name="step_chi512_k2", kind="step", chi=512, k=2, clusters=4, precision="fp32",
             spectrum="decaying", decades=8.0, cutoff=1e-12, ragged=True),
        # the chi_max = 1024 configuration: a steep spectrum, the cutoff decides the rank
        dict(name="step_chi1024_k2_steep", kind="step", chi=1024, k=2, clusters=2, precision="fp32",
             spectrum="decaying", decades=20.0, cutoff=1e-8, ragged=False),
        # the chi_max = 1024 configuration at saturation: a flat spectrum, chi_max decides the rank
        dict(name="step_chi1024_k2_saturated", kind="step", chi=1024, k=2, clusters=4, precision="fp32",
             spectrum="flat", decades=0.0, cutoff=1e-8, ragged=False),
        # a whole exact run in complex128 (12 qubits, 10 layers)
        dict(name="circuit_n12_exact_fp64", kind="circuit", n=12, layers=10, chi_max=64, k_max=4,
             cutoff=0.0, t_share=1 / 3, precision="fp64"),
        # a whole run of the chi_max = 256 configuration's circuit family (100 qubits, 20 layers)
        dict(name="circuit_n100_clifford_t", kind="circuit", n=100, layers=20, chi_max=256, k_max=6,
             cutoff=1e-10, t_share=0.1, precision="fp32"),
        # amplitudes of a stored 100-qubit state
        dict(name="amplitude_n100_chi256", kind="amplitude", n=100, chi=256, count=4, precision="fp32"),
        # the allocation-free two-site split inside another program's loop
        dict(name="split2_chi48x64", kind="split2", chi_l=48, chi_r=64, chi_max=64, decades=8.0, cutoff=1e-8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["circuit", "amplitude", "split2"])
    if kind == "circuit":
        n = rng.randint(10, 100)
        exact = n <= 16 and rng.random() < 0.5
        return dict(kind=kind, n=n, layers=rng.randint(8, 20), chi_max=64 if exact else 256,
                    k_max=rng.randint(3, 6), cutoff=0.0 if exact else 1e-10,
                    t_share=round(rng.uniform(0.05, 0.33), 3), precision="fp64" if exact else "fp32")
    if kind == "amplitude":
        return dict(kind=kind, n=_log_int(rng, 16, 200), chi=_log_int(rng, 8, 512), count=rng.randint(1, 8),
                    precision=rng.choice(["fp32", "fp32", "fp64"]))
    if kind == "split2":
        return dict(kind=kind, chi_l=_log_int(rng, 4, 128), chi_r=_log_int(rng, 4, 128),
                    chi_max=_log_int(rng, 16, 128), decades=round(rng.uniform(5.0, 10.0), 2), cutoff=1e-8)
    fp64 = rng.random() < 0.15
    chi = _log_int(rng, 4, 96 if fp64 else 1024)
    k = 2 if chi > 512 else rng.randint(2, 3) if chi > 128 else rng.randint(2, 4)
    flat = rng.random() < 0.25
    k = 2 if flat else k
    most = max(1, min(16, int(2.0e9 / (chi ** 3 * (k - 1)))))
    return dict(kind=kind, chi=chi, k=k, clusters=rng.randint(1, most), precision="fp64" if fp64 else "fp32",
                spectrum="flat" if flat else "decaying", decades=0.0 if flat else round(rng.uniform(6.0, 12.0), 2),
                cutoff=rng.choice([1e-8, 1e-10]), ragged=rng.random() < 0.6)


# ---- inputs ------------------------------------------------------------------
def _dtype(case):
    return torch.complex128 if case.get("precision") == "fp64" else torch.complex64


def _weights(case, n, rng):
    """Schmidt values of a bond: geometric decay with scatter, or Porter-Thomas (saturated)."""
    if case.get("spectrum") == "flat":
        w = np.sort(rng.exponential(1.0, size=n))[::-1]
    else:
        w = 10.0 ** (-case["decades"] * np.arange(n) / n) * rng.uniform(0.8, 1.2, size=n)
        w = np.sort(w)[::-1]
    return np.sqrt(w / w.sum())


def _isometry(rows, cols, gen, dtype):
    """A random right isometry (rows <= cols, orthonormal rows) on the device."""
    g = torch.randn(cols, rows, dtype=dtype, device="cuda", generator=gen)
    return torch.linalg.qr(g)[0].conj().resolve_conj().transpose(0, 1).contiguous()


def _state(case, chis, seed):
    """Sites and spectra of a random right-canonical state with the given bonds."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    sites = [_isometry(chis[q], 2 * chis[q + 1], gen, _dtype(case)).reshape(chis[q], 2, chis[q + 1])
             for q in range(len(chis) - 1)]
    lams = [torch.from_numpy(_weights(case, c, rng)).cuda() for c in chis]
    return sites, lams


def _random_gates(n, layers, t_share, p1, p2, rng):
    """Random layers of CNOT / CZ on neighbours and H, S, T on the free qubits, as gate rows."""
    rows = []
    kinds, share = [T, H, S], [t_share, (1 - t_share) / 2, (1 - t_share) / 2]
    for _ in range(layers):
        q = 0
        while q < n:
            if q + 1 < n and rng.random() < p2:
                rows.append((2, q, q + 1, -1, int(rng.choice([CNOT, CZ]))))
                q += 2
                continue
            if rng.random() < p1:
                rows.append((1, q, -1, -1, int(rng.choice(kinds, p=share))))
            q += 1
    return np.array(rows, dtype=np.int32).reshape(-1, 5)


def _step_chis(case, rng):
    """Bond dimensions of a chain that holds the clusters side by side: ramps of powers of two at
    both ends, chi (or, ragged, 3/4 chi to chi) in between."""
    chi, k = case["chi"], case["k"]
    ramp = []
    while len(ramp) == 0 or 2 * ramp[-1] < chi:
        ramp.append(2 * ramp[-1] if ramp else 1)
    inner = [chi if not case["ragged"] else int(rng.integers(max(2, (3 * chi + 3) // 4), chi + 1))
             for _ in range(case["clusters"] * k + 1)]
    return ramp + inner + ramp[::-1], len(ramp)


def _step_parts(case, seed):
    chis, q0 = _step_chis(case, np.random.default_rng(case["chi"] * 31 + case["clusters"]))
    rng = np.random.default_rng(seed + 1)
    sites, lams = _state(case, chis, seed)
    clusters, Us = [], []
    for i in range(case["clusters"]):
        k = case["k"]
        # layers of Haar-random two-site gates, as an iteration's layers contract to
        U = np.eye(2 ** k, dtype=np.complex128)
        for layer in range(2):
            for b in range(layer % 2 if k > 2 else 0, k - 1, 2):
                g = np.linalg.qr(rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4)))[0]
                U = np.kron(np.kron(np.eye(2 ** b), g), np.eye(2 ** (k - b - 2))) @ U
        clusters.append((q0 + i * k, k))
        Us.append(U)
    return chis, sites, lams, clusters, Us


def _config(case, n, chi, k):
    prec = P.FP64 if case["precision"] == "fp64" else P.FP32
    return P.make_config(n, chi, case["cutoff"], k + 2 * math.ceil(math.log2(max(chi, 2))), 0, k, prec)


def _bits(count, n, seed):
    rng = np.random.default_rng(seed + 2)
    return [rng.integers(0, 2, n).astype(np.uint8) for _ in range(count)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        chis, sites, lams, where, Us = _step_parts(case, seed)
        cfg = _config(case, len(chis) - 1, max(chis), case["k"])
        torch.cuda.synchronize()
        return dict(case=case, chis=np.array(chis, dtype=np.int32), sites=sites, lams=lams,
                    site_ptrs=[s.data_ptr() for s in sites], lam_ptrs=[x.data_ptr() for x in lams],
                    lam_host=[lams[q].cpu().numpy() for q, _ in where],
                    clusters=[P.Cluster(q, k, 0, 0) for q, k in where], Us=Us, mps=P.MPS(cfg),
                    read=torch.empty((case["k"], 4 * max(chis) ** 2), dtype=torch.float64).pin_memory())
    if kind == "circuit":
        rng = np.random.default_rng(seed)
        rows = _random_gates(case["n"], case["layers"], case["t_share"], 0.5, 0.3, rng)
        # a last layer of X^(1/4) on every qubit, after which no bit string is out of reach
        rows = np.concatenate([rows, np.array([(1, q, -1, -1, X14) for q in range(case["n"])], dtype=np.int32)])
        return dict(case=case, circuit=P.Circuit(case["n"], rows, np.zeros(len(rows))), rows=rows,
                    cfg=_config(case, case["n"], case["chi_max"], case["k_max"]), bits=_bits(4, case["n"], seed))
    if kind == "amplitude":
        n = case["n"]
        chis = [min(case["chi"], 2 ** min(b, n - b, 30)) for b in range(n + 1)]
        sites, lams = _state(dict(case, spectrum="flat"), chis, seed)
        mps = P.MPS(_config(dict(case, cutoff=0.0), n, case["chi"], 2))
        torch.cuda.synchronize()
        mps.load_device(np.array(chis, dtype=np.int32), [s.data_ptr() for s in sites],
                        [x.data_ptr() for x in lams])
        return dict(case=case, mps=mps, sites=sites, bits=_bits(case["count"], n, seed))
    # split2: theta of two random isometries, as after a two-site gate
    cl, cr = case["chi_l"], case["chi_r"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    theta = torch.randn(cl, 4, cr, dtype=torch.complex64, device="cuda", generator=gen) / math.sqrt(4 * cr)
    lam = torch.from_numpy(_weights(case, cl, np.random.default_rng(seed))).cuda()
    most = min(case["chi_max"], 2 * cl, 2 * cr)
    left = torch.zeros(cl * 2 * most, dtype=torch.complex64, device="cuda")
    right = torch.zeros(most * 2 * cr, dtype=torch.complex64, device="cuda")
    spec = torch.zeros(most, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return dict(case=case, theta=theta, lam=lam, left=left, right=right, spec=spec)


# ---- one pass ----------------------------------------------------------------
def _theta(lam, sites):
    """diag(lam) B_q B_{q+1} ... of torch tensors or numpy arrays, as a matrix."""
    a = sites[0].shape[0]
    t = (lam[:, None] * sites[0].reshape(a, -1)).reshape(-1, sites[0].shape[2])
    for s in sites[1:]:
        t = (t @ s.reshape(s.shape[0], -1)).reshape(-1, s.shape[2])
    return t


def _read_theta(state, chi, i):
    """The theta of the i-th updated cluster: on the host for narrow bonds, else on the device."""
    case, c = state["case"], state["clusters"][i]
    host = case["chi"] <= 64
    sites = []
    for j in range(c.k):
        a, b = int(chi[c.q0 + j]), int(chi[c.q0 + j + 1])
        buf = state["read"][j]
        rc = P.lib.mps_to_host(state["mps"]._h, c.q0 + j,
                               ctypes.cast(buf.data_ptr(), ctypes.POINTER(ctypes.c_double)), buf.numel())
        if rc != P.OK:
            raise P.CtebdError(P.last_error())
        if host:
            sites.append(buf.numpy()[:4 * a * b].view(np.complex128).reshape(a, 2, b))
        else:
            sites.append(torch.view_as_complex(buf[:4 * a * b].view(-1, 2)).cuda(non_blocking=True)
                         .to(_dtype(case)).view(a, 2, b))
    if host:
        return _in_precision(case, _theta(state["lam_host"][i], sites)).reshape(-1)
    torch.cuda.current_stream().synchronize()  # the host buffers are used again
    return torch.view_as_real(_theta(state["lams"][c.q0].to(_dtype(case)), sites)).reshape(-1)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        mps, clusters = state["mps"], state["clusters"]
        mps.load_device(state["chis"], state["site_ptrs"], state["lam_ptrs"])
        f = mps.step(clusters, state["Us"])
        chi = mps.bond_dims()
        spectra = _padded([mps.lam(c.q0 + j) for c in clusters for j in range(1, c.k)], int(max(state["chis"])))
        out = dict(chi=chi, f=_in_precision(case, f), spectra=_in_precision(case, spectra))
        if case["spectrum"] != "flat":
            # in a flat spectrum the cut falls among nearly equal weights, and which of two such directions
            # is kept is a matter of rounding: the updated sites are no result there that could be compared
            thetas = [_read_theta(state, chi, i) for i in range(len(clusters))]
            out["theta"] = np.concatenate(thetas) if case["chi"] <= 64 else torch.cat(thetas)
        return out
    if kind == "circuit":
        mps = P.simulate(state["circuit"], state["cfg"])
        amps = np.array([mps.amplitude(b) for b in state["bits"]])
        return dict(amplitudes=_in_precision(case, amps), chi=mps.bond_dims(),
                    f=_in_precision(case, np.array([mps.fidelity()])))
    if kind == "amplitude":
        return dict(amplitudes=_in_precision(case, np.array([state["mps"].amplitude(b) for b in state["bits"]])))
    cl, cr = case["chi_l"], case["chi_r"]
    r, f = P.split2_noalloc(state["theta"].data_ptr(), state["lam"].data_ptr(), cl, cr, case["chi_max"],
                            case["cutoff"], state["left"].data_ptr(), state["right"].data_ptr(),
                            state["spec"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    theta = _theta(state["lam"].to(torch.complex64),
                   [state["left"][:cl * 2 * r].view(cl, 2, r), state["right"][:r * 2 * cr].view(r, 2, cr)])
    return dict(theta=torch.view_as_real(theta), r=r, f=np.float32(f),
                spectrum=torch.nn.functional.pad(state["spec"][:r].float(), (0, state["spec"].numel() - r)))


def _padded(spectra, n):
    """Spectra of any rank as rows of n values."""
    out = np.zeros((len(spectra), n))
    for row, s in zip(out, spectra):
        row[:len(s)] = s
    return out


def _in_precision(case, a):
    """Host copies come in 64 bits whatever the mode: results of the FP32 mode in the type they carry."""
    if case["precision"] == "fp64":
        return a
    return a.astype(np.complex64 if np.iscomplexobj(a) else np.float32)


# ---- what a pass cannot do without --------------------------------------------
def _svd_flops(m, n):
    """A thin complex SVD through the Gram matrix of the narrow side: Gram, eigenvectors, projection."""
    a, b = max(m, n), min(m, n)
    return 8.0 * a * b * b + 8.0 * (4 / 3 + 2) * b ** 3 + 8.0 * a * b * b


def work(case):
    kind = case["kind"]
    esz = 16 if case.get("precision") == "fp64" else 8
    if kind == "step":
        chi, k = case["chi"] * (0.875 if case["ragged"] else 1.0), case["k"]
        per = 8.0 * 4 ** k * chi * chi
        for j in range(1, k):
            per += 8.0 * chi * 2 ** j * chi * 2 * chi
            per += _svd_flops(chi * 2 ** j, 2 * chi)
        site = 2 * chi * chi * esz
        return {"bytes": case["clusters"] * (2 * k * site + 2 * 2 ** k * chi * chi * esz), "flops": case["clusters"] * per}
    if kind == "circuit":
        gates = case["n"] * case["layers"] * 0.5
        return {"bytes": gates * 2 * 64 * esz, "flops": gates * (_svd_flops(8, 8) + 8 * 8 ** 3)}
    if kind == "amplitude":
        n, chi = case["n"], case["chi"]
        dims = [min(chi, 2 ** min(b, n - b, 30)) for b in range(n + 1)]
        e = sum(dims[q] * dims[q + 1] for q in range(n))
        return {"bytes": case["count"] * e * esz, "flops": case["count"] * 8.0 * e}
    cl, cr = case["chi_l"], case["chi_r"]
    r = min(case["chi_max"], 2 * cl, 2 * cr)
    return {"bytes": 8.0 * (4 * cl * cr + 2 * r * (cl + cr)), "flops": _svd_flops(2 * cl, 2 * cr)}


# ---- the same in 64 bits ---------------------------------------------------------
def _split64(m, w, chi_max, cutoff, floor):
    """One truncated split of the rows-weighted matrix: (site, remainder, spectrum, f)."""
    u, s, vh = np.linalg.svd(w[:, None] * m, full_matrices=False)
    p = s * s
    total = p.sum()
    tail = np.append(np.cumsum(p[::-1])[::-1][1:], 0.0)
    r = len(p)
    if cutoff > 0:
        r = int(np.argmax(tail <= cutoff * total)) + 1
    r = max(1, min(r, int((p > floor * floor * p[0]).sum()), chi_max))
    kept = p[:r].sum()
    return vh[:r], (m @ vh[:r].conj().T) / math.sqrt(kept), np.sqrt(p[:r] / kept), kept / total


def _exact_step(case, seed):
    chis, sites, lams, where, Us = _step_parts(case, seed)
    k, chi_max = case["k"], max(chis)
    if len(where) * sum((2 * chi_max) ** 2 * min(2 ** j, 4) * chi_max for j in range(1, k)) > 6e9:
        return None
    floor = 1e-13 if case["precision"] == "fp64" else 1e-6
    thetas, fs, spectra = [], [], []
    for (q0, _), U in zip(where, Us):
        a, b = chis[q0], chis[q0 + k]
        t = sites[q0].to(torch.complex128).cpu().numpy().reshape(a * 2, -1)
        for j in range(1, k):
            s = sites[q0 + j].to(torch.complex128).cpu().numpy()
            t = (t @ s.reshape(s.shape[0], -1)).reshape(-1, s.shape[2])
        t = np.einsum("st,atb->asb", U, t.reshape(a, 2 ** k, b))
        lam = lams[q0].cpu().numpy()
        new, out, mine = [], [], []
        rem, right = t, b
        for j in range(k - 1, 0, -1):
            site, rem, spec, f = _split64(rem.reshape(a * 2 ** j, 2 * right), np.repeat(lam, 2 ** j), chi_max,
                                          case["cutoff"], floor)
            new.insert(0, site.reshape(len(spec), 2, right))
            mine.append(f)
            out.insert(0, spec)
            right = len(spec)
        t = _theta(lam, [rem.reshape(a, 2, right)] + new)
        thetas.append(np.ascontiguousarray(t).reshape(-1).view(np.float64))
        fs += mine
        spectra += out
    out = dict(chi=None, f=np.array(fs), spectra=_padded(spectra, chi_max))
    if case["spectrum"] != "flat":
        out["theta"] = np.concatenate(thetas)
    return out


def _exact_circuit(case, seed):
    st = prepare(case, seed)
    n = case["n"]
    if n > 18:
        return None
    r2 = math.sqrt(0.5)
    w = complex(r2, r2)
    one = {H: np.array([[r2, r2], [r2, -r2]]), S: np.diag([1, 1j]), T: np.diag([1, w]),
           X14: np.array([[1 + w, 1 - w], [1 - w, 1 + w]]) / 2}
    two = {CNOT: np.eye(4)[[0, 1, 3, 2]], CZ: np.diag([1, 1, 1, -1])}
    psi = np.zeros(2 ** n, dtype=np.complex128)
    psi[0] = 1
    for nq, a, _, _, kind in st["rows"]:
        g = (one if nq == 1 else two)[int(kind)]
        psi = np.einsum("st,atb->asb", g, psi.reshape(2 ** int(a), 2 ** int(nq), -1)).reshape(-1)
    amps = [psi[int("".join(map(str, b)), 2)] for b in st["bits"]]
    return dict(amplitudes=np.array(amps), chi=None, f=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "circuit":
        return _exact_circuit(case, seed)
    if kind == "amplitude":
        st = prepare(case, seed)
        out = []
        for bits in st["bits"]:
            v = torch.ones(1, 1, dtype=torch.complex128, device="cuda")
            for s, x in zip(st["sites"], bits):
                v = v @ s[:, int(x), :].to(torch.complex128)
            out.append(v.item())
        return dict(amplitudes=np.array(out))
    st = prepare(case, seed)
    cl, cr = case["chi_l"], case["chi_r"]
    m = st["theta"].to(torch.complex128).cpu().numpy().reshape(2 * cl, 2 * cr)
    w = np.repeat(st["lam"].cpu().numpy(), 2)
    site, rem, spec, f = _split64(m, w, min(case["chi_max"], 2 * cl, 2 * cr), case["cutoff"], 1e-6)
    theta = np.ascontiguousarray((w[:, None] * rem) @ site)
    return dict(theta=theta.reshape(-1).view(np.float64).reshape(-1, 2), r=None, f=np.array([f]),
                spectrum=_padded([spec], min(case["chi_max"], 2 * cl, 2 * cr))[0])
