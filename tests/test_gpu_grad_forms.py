"""The VMC gradient of each 16-bit form (Eq. grad_def), measured per result:
the form samples its own set, computes its local energies and statistics and
then its gradient, all through the library; the FP64 oracle computes the
gradient on the same samples and counts from its own local energies.

The 16-bit forms take log psi's adjoint from the FP32 kernels of the same
parameters, so the two gradients differ by the FP32 adjoint's rounding and by
the 16-bit local energies entering the cotangents 2 w (E_loc - E).  With a
per-sample local-energy deviation delta and a spread sigma of E_loc - E, the
relative error of the cotangents is about delta / sigma; the bar is a relative
L2 error of 1e-3."""
import numpy as np
import pytest
import torch

from oracle.anqs import MLPAnsatz, TFAnsatz
from oracle.hamiltonian import Hamiltonian as OHam
from oracle.sector import molecular_isphys
from oracle.vmc import energy_stats, gradient, local_energy
from synthetic import workload

pytestmark = pytest.mark.gpu
BAR = 1e-3


@pytest.fixture(scope="module")
def A():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_04166_gb300 as mod
    from paper_2310_04166_gb300 import _lib
    _lib.load()
    return mod


def _problem(A, name):
    w = workload(name, bias_std=0.2)
    ham = A.Hamiltonian(w["h"], w["g"], w["e_nuc"], w["n_alpha"], w["n_beta"])
    params = torch.tensor(w["params"], device="cuda")
    if w["kind"] == "mlp":
        model = A.Model.mlp(w["n"], w["width"], w["n_hidden"], params, "bf16")
        om = MLPAnsatz(w["params_struct"], w["n"])
    else:
        model = A.Model.transformer(w["n"], w["d_model"], w["n_heads"], w["n_layers"], params, "bf16")
        om = TFAnsatz(w["params_struct"], w["n"], w["n_heads"])
    ip = molecular_isphys(w["n"], w["n_alpha"], w["n_beta"])
    oham = OHam(w["h"], w["g"], w["e_nuc"], w["n_alpha"], w["n_beta"])
    return w, ham, model, om, ip, oham


@pytest.mark.parametrize("name,Ns,keep", [("h2o", 100_000, None), ("n2", 20_000, 64)])
def test_16bit_form_gradient_against_oracle(A, name, Ns, keep):
    """h2o: the whole unique set of one N_s = 1e5 pass.  n2: the 64 most
    frequent samples of one N_s = 2e4 pass (the oracle's transformer local
    energy is too slow for the whole set within a test)."""
    w, ham, model, om, ip, oham = _problem(A, name)
    x, c = A.sample(model, ham, Ns, seed=21)
    if keep is not None:
        order = torch.argsort(c.cpu(), descending=True, stable=True)[:keep].to(x.device)
        x, c = x[order].contiguous(), c[order].contiguous()
    ere, eim, stats = A.local_energy(model, ham, x, c)
    g = A.grad(model, ham, x, c, ere, eim, stats).cpu().numpy().astype(np.float64)
    assert model.status() == 0

    xs, cs = x.cpu().numpy().astype(np.uint64), c.cpu().numpy()
    e_ref = local_energy(om, ip, oham, xs)
    s_ref = energy_stats(e_ref, cs)
    g_ref = np.concatenate([t.reshape(-1).numpy() for t in gradient(om, ip, xs, cs, e_ref, s_ref)])
    rel = np.linalg.norm(g - g_ref) / np.linalg.norm(g_ref)
    d = np.abs(ere.cpu().numpy() - e_ref.real)
    assert rel < BAR, (rel, d.max(), np.sqrt(s_ref[2]))


def _batch_problem(A, k, n_samples):
    from synthetic import batch32_problem, flatten_mlp, mlp_params
    p = batch32_problem(k)
    ham = A.Hamiltonian(p["h"], p["g"], p["e_nuc"], p["n_alpha"], p["n_beta"])
    P = mlp_params(p["seed"], p["n"], p["width"], p["n_hidden"], 0.2)
    model = A.Model.mlp(p["n"], p["width"], p["n_hidden"], torch.tensor(flatten_mlp(P), device="cuda"), "bf16")
    om = MLPAnsatz(P, p["n"])
    ip = molecular_isphys(p["n"], p["n_alpha"], p["n_beta"])
    oham = OHam(p["h"], p["g"], p["e_nuc"], p["n_alpha"], p["n_beta"])
    return ham, model, om, ip, oham


@pytest.mark.parametrize("case", ["h2o", "batch14", "batch0"])
def test_tensor_core_adjoint_against_oracle(A, case):
    """The 16-bit MLP's adjoint (tcgen05, fp16 operands, per-tile scaled
    cotangents) with the oracle's own local energies as input, so that only
    the adjoint's arithmetic differs: relative L2 error below 5e-4 (the CPU
    emulation of its rounding gives about 2e-4 on h2o).  h2o: 441 rows, four
    tiles, the last one partial; problem 14 of the 32-problem workload (7
    orbitals); problem 0 (12 orbitals, 10+10 electrons: the widest layer-1
    input the kernel takes)."""
    if case == "h2o":
        w, ham, model, om, ip, oham = _problem(A, "h2o")
        Ns = 100_000
    else:
        ham, model, om, ip, oham = _batch_problem(A, int(case[5:]), 20_000)
        Ns = 20_000
    x, c = A.sample(model, ham, Ns, seed=31)
    if x.numel() > 600:
        order = torch.argsort(c.cpu(), descending=True, stable=True)[:600].to(x.device)
        x, c = x[order].contiguous(), c[order].contiguous()
    xs, cs = x.cpu().numpy().astype(np.uint64), c.cpu().numpy()
    e_ref = local_energy(om, ip, oham, xs)
    s_ref = energy_stats(e_ref, cs)
    g = A.grad(model, ham, x, c, torch.tensor(e_ref.real, device="cuda"), torch.tensor(e_ref.imag, device="cuda"),
               torch.tensor(s_ref, device="cuda")).cpu().numpy().astype(np.float64)
    assert model.status() == 0
    g_ref = np.concatenate([t.reshape(-1).numpy() for t in gradient(om, ip, xs, cs, e_ref, s_ref)])
    rel = np.linalg.norm(g - g_ref) / np.linalg.norm(g_ref)
    assert rel < 5e-4, rel
    # every parameter block is written: slot 0's first-layer bias and the heads too
    assert np.isfinite(g).all()


def test_tensor_core_adjoint_with_device_row_count(A):
    """The bench's shape: capacity rows on the host, the unique count on the
    device; tiles past the count contribute nothing."""
    w, ham, model, om, ip, oham = _problem(A, "h2o")
    x, c = A.sample(model, ham, 100_000, seed=32)
    k = x.numel()
    cap = k + 300
    xb = torch.zeros(cap, dtype=torch.int64, device="cuda")
    cb = torch.zeros(cap, dtype=torch.int64, device="cuda")
    xb[:k], cb[:k] = x, c
    ere, eim, st = A.local_energy(model, ham, x, c)
    erb = torch.zeros(cap, dtype=torch.float64, device="cuda")
    eib = torch.zeros(cap, dtype=torch.float64, device="cuda")
    erb[:k], eib[:k] = ere, eim
    g1 = A.grad(model, ham, x, c, ere, eim, st)
    nd = torch.tensor([k], dtype=torch.int64, device="cuda")
    g2 = A.grad(model, ham, xb, cb, erb, eib, st, n_dev=nd)
    assert torch.equal(g1, g2)


def test_tensor_core_adjoint_directly_after_a_repack(A):
    """The adjoint kernel bulk-copies the packed weight images before its
    dependency wait.  The packing kernel never lets a dependent launch start
    early, so a gradient queued directly after a repack (no other kernel in
    between: preallocated output and workspace) sees the new weights."""
    w, ham, model, om, ip, oham = _problem(A, "h2o")
    x, c = A.sample(model, ham, 100_000, seed=34)
    ere, eim, st = A.local_energy(model, ham, x, c)
    ws = A._ws(A.grad_workspace_bytes(model, ham, x.numel()), x.device)
    g1 = torch.empty(model.n_params, dtype=torch.float32, device=x.device)
    g2 = torch.empty_like(g1)
    model.params.mul_(1.25)
    torch.cuda.synchronize()
    model.sync()
    A.grad(model, ham, x, c, ere, eim, st, workspace=ws, out=g1)
    torch.cuda.synchronize()
    A.grad(model, ham, x, c, ere, eim, st, workspace=ws, out=g2)
    torch.cuda.synchronize()
    assert model.status() == 0
    assert torch.equal(g1, g2)


def _adjoint_problem(A, n, na, nb, hidden, m, seed, width=128, form="bf16"):
    """A 16-bit MLP, m random determinants of the sector and random local energies."""
    from synthetic import flatten_mlp, integrals, mlp_params
    h, g, e = integrals(seed, n, 2)
    ham = A.Hamiltonian(h, g, e, na, nb)
    P = mlp_params(seed, n, width, hidden, 0.2)
    model = A.Model.mlp(n, width, hidden, torch.tensor(flatten_mlp(P), device="cuda"), form)
    rng = np.random.default_rng(seed)
    occ = lambda k: (np.argsort(rng.random((m, n)), axis=1)[:, :k]).astype(np.uint64)
    x = (np.uint64(1) << (np.uint64(2) * occ(na))).sum(1, dtype=np.uint64)
    x = x + (np.uint64(2) << (np.uint64(2) * occ(nb))).sum(1, dtype=np.uint64)
    return ham, P, model, x, rng


def _grad_and_kernels(A, model, ham, x, cnt, e, stats):
    """The gradient, and how often the tensor-core adjoint's kernel ran."""
    import ctypes as C
    from paper_2310_04166_gb300 import _lib
    lib = _lib.load()
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    _lib.check(lib.anqs_profile_enable(1))
    g = A.grad(model, ham, t(x.astype(np.int64)), t(cnt.astype(np.int64)), t(e.real), t(e.imag), t(stats))
    torch.cuda.synchronize()
    ran, k = {}, 0
    while True:
        name, c, ms = C.c_char_p(), C.c_uint64(), C.c_double()
        if lib.anqs_profile_read(k, C.byref(name), C.byref(c), C.byref(ms)) != 0:
            break
        ran[name.value.decode()] = c.value
        k += 1
    _lib.check(lib.anqs_profile_enable(0))
    return g.cpu().numpy().astype(np.float64), ran["mlp_tc_grad_kernel"]


def _adjoint_reference(P, n, na, nb, x, cnt, e, stats):
    """The FP64 oracle's gradient for given local energies and statistics."""
    g = gradient(MLPAnsatz(P, n), molecular_isphys(n, na, nb), x, cnt, e, stats)
    return np.concatenate([t.reshape(-1).numpy() for t in g])


@pytest.mark.parametrize("n,na,nb", [(17, 3, 2), (18, 3, 3), (26, 2, 3), (32, 2, 1)])
@pytest.mark.parametrize("hidden", [1, 2])
def test_tensor_core_adjoint_of_wide_inputs(A, n, na, nb, hidden):
    """Layer-1 inputs of 64 to 128 columns (17 to 32 orbitals) run on the
    tensor cores with one and two hidden layers, two tiles, the last one
    partial; the module's bar."""
    ham, P, model, x, rng = _adjoint_problem(A, n, na, nb, hidden, 200, 11 * n + hidden)
    cnt = rng.integers(1, 50, size=x.size)
    e = rng.normal(size=x.size) + 1j * rng.normal(size=x.size)
    stats = energy_stats(e, cnt)
    g, ran = _grad_and_kernels(A, model, ham, x, cnt, e, stats)
    ref = _adjoint_reference(P, n, na, nb, x, cnt, e, stats)
    assert ran == 1 and model.status() == 0
    assert np.linalg.norm(g - ref) < BAR * np.linalg.norm(ref)


def _tensors(x, cnt, e):
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    return t(x.astype(np.int64)), t(cnt.astype(np.int64)), t(e.real), t(e.imag)


@pytest.mark.parametrize("hidden", [2, 3])
def test_tensor_core_adjoint_keeps_small_rows_beside_a_large_one(A, hidden):
    """One sample holds nearly all draws (1e7 of them, alone in its tile), 29
    tiles of samples drawn once follow, several tiles per CTA.  The columns of
    W_1 of outcomes that the large sample does not take get their gradient
    from the others alone: as without it, up to the order of float32 sums
    (3,712 rows: some 1e-6 of a column block's norm; the bar is 1e-5)."""
    n, na, nb = 12, 6, 6
    ham, P, model, x, rng = _adjoint_problem(A, n, na, nb, hidden, 30 * 128, 5 + hidden)
    cnt = np.ones(x.size, dtype=np.int64)
    cnt[1:128] = 0
    cnt[0] = 10_000_000
    e = rng.normal(size=x.size) + 1j * rng.normal(size=x.size)
    stats = np.array([0.3, -0.2, 1.0, float(cnt.sum())])
    st = torch.tensor(stats, device="cuda")
    without = cnt.copy()
    without[0] = 0
    g, g0 = (A.grad(model, ham, *_tensors(x, c, e), st).cpu().numpy().astype(np.float64) for c in (cnt, without))
    assert model.status() == 0
    off = 0
    for p, layers in enumerate(P):
        for k, (w, b) in enumerate(layers):
            if k == 0 and p:
                v = (int(x[0]) >> (2 * np.arange(p))) & 3
                others = np.ones(4 * p, dtype=bool)
                others[4 * np.arange(p) + v] = False
                a, r = (u[off:off + w.size].reshape(w.shape)[:, others] for u in (g, g0))
                assert np.linalg.norm(a - r) <= 1e-5 * np.linalg.norm(r), p
            off += (w.size if w is not None else 0) + b.size


@pytest.mark.parametrize("hidden,tiles", [(2, 26), (3, 26), (2, 200), (3, 200)])
def test_tensor_core_adjoint_with_several_tiles_per_cta(A, hidden, tiles):
    """2 to 3 tiles per CTA, and more than the 16 after which a CTA writes its
    sums (12 CTAs per slot at 12 orbitals), the last tile partial: against the
    oracle at the module's bar, and against the FP64 sum of calls of one tile
    each (float32 sums of at most 150 terms in another order: 150 / 2^24 =
    9e-6 at worst, the bar is twice that).  Then the same buffers with a device
    row count that leaves some CTAs without a tile: as a call of those rows."""
    n, na, nb = 12, 6, 6
    ham, P, model, x, rng = _adjoint_problem(A, n, na, nb, hidden, 390, 17 + hidden)
    cnt = rng.integers(1, 40, size=x.size)
    e = rng.normal(size=x.size) + 1j * rng.normal(size=x.size)
    rep = tiles * 128 // x.size
    stats = energy_stats(e, cnt)
    stats[3] *= rep
    X, N, R, I = _tensors(np.tile(x, rep), np.tile(cnt, rep), np.tile(e, rep))
    assert X.numel() % 128 and -(-X.numel() // 128) > 2 * 12
    st = torch.tensor(stats, device="cuda")
    g = A.grad(model, ham, X, N, R, I, st)
    ref = _adjoint_reference(P, n, na, nb, x, cnt * rep, e, stats)
    assert np.linalg.norm(g.cpu().numpy() - ref) < BAR * np.linalg.norm(ref)
    parts = torch.zeros(model.n_params, dtype=torch.float64, device="cuda")
    for k in range(0, X.numel(), 128):
        s = slice(k, k + 128)
        parts += A.grad(model, ham, X[s].contiguous(), N[s].contiguous(), R[s].contiguous(), I[s].contiguous(),
                        st).double()
    assert torch.linalg.norm(g.double() - parts) <= 1.8e-5 * torch.linalg.norm(parts)
    few = 700  # six tiles for twelve CTAs
    nd = torch.tensor([few], dtype=torch.int64, device="cuda")
    a = A.grad(model, ham, X, N, R, I, st, n_dev=nd)
    b = A.grad(model, ham, *(t[:few].contiguous() for t in (X, N, R, I)), st)
    assert torch.equal(a, b) and model.status() == 0
