"""Local energies over distinct connected determinants (csrc/eloc_unique.cu).

The FP32 forms are compared with the static-scratch entry point, which
evaluates every connected determinant by itself through the same assembly:
the results are equal bit for bit.  The 16-bit and NADE forms are compared
with the sum over anqs_connected's list and anqs_logpsi's amplitudes: the same
terms added in another order, so each log-amplitude differs by float32
rounding (n sums of values below about 20: 2e-5), and E_loc by that times the
sum of |H psi'/psi|.
"""
import ctypes as C
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    import paper_2310_04166_gb300 as A
    return A


def _problem(A, kind, form, n, na, nb, seed, z2=False, du=0):
    from synthetic import (flatten_mlp, flatten_nade, flatten_tf, integrals, integrals_z2, mlp_params, nade_params,
                           tf_params, z2_qubit_masks)
    labels = [p % 2 for p in range(n)]
    h, g, e = integrals_z2(seed, n, 2 * n, labels) if z2 else integrals(seed, n, 2 * n)
    ham = A.Hamiltonian(h, g, e, na, nb)
    if z2:
        ham.set_z2(z2_qubit_masks(labels))
    if du:
        ham.set_pruning(du)
    t = lambda a: torch.tensor(a, device="cuda")
    if kind == "mlp":
        return A.Model.mlp(n, 64, 2, t(flatten_mlp(mlp_params(seed, n, 64, 2, 0.2))), form), ham
    if kind == "nade":
        return A.Model.nade(n, 32, t(flatten_nade(nade_params(seed, n, 32, 0.1)))), ham
    return A.Model.transformer(n, 64, 4, 1, t(flatten_tf(tf_params(seed, n, 64, 1, 0.1))), form), ham


def _dets(n, na, nb, m, seed, parity=None):
    rng = np.random.default_rng(seed)
    out = set()
    for _ in range(50 * m):
        x = sum(1 << (2 * int(p)) for p in rng.choice(n, na, replace=False))
        x += sum(1 << (2 * int(p) + 1) for p in rng.choice(n, nb, replace=False))
        if parity is None or bin(x & parity[0]).count("1") % 2 == parity[1]:
            out.add(x - ((x >> 63) << 64))  # as int64
        if len(out) == m:
            break
    return torch.tensor(sorted(out), dtype=torch.int64, device="cuda")


def _static(A, model, ham, x, cnt):
    from paper_2310_04166_gb300 import _lib
    ere, eim = (torch.empty(x.numel(), dtype=torch.float64, device="cuda") for _ in range(2))
    st = torch.empty(4, dtype=torch.float64, device="cuda")
    _lib.check(_lib.load().anqs_local_energy_static(model._m, ham.handle, x.data_ptr(), cnt.data_ptr(), x.numel(),
                                                    ere.data_ptr(), eim.data_ptr(), st.data_ptr(),
                                                    C.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return ere, eim, st


# (n, na, nb, samples): one orbital, full shells (no excitations), few samples of a larger sector (bitmap, samples
# split over CTAs), most of a small sector (all prefixes), odd counts, several bitmap blocks
SHAPES = [(1, 1, 0, 1), (3, 3, 0, 1), (4, 2, 2, 36), (5, 1, 4, 3), (7, 5, 2, 9), (9, 4, 5, 33), (10, 5, 5, 130)]


@pytest.mark.parametrize("kind", ["mlp", "tf"])
@pytest.mark.parametrize("n,na,nb,m", SHAPES)
@pytest.mark.parametrize("z2,du", [(False, 0), (True, 0), (False, 1)])
def test_fp32_equals_every_determinant_by_itself(A, kind, n, na, nb, m, z2, du):
    model, ham = _problem(A, kind, "fp32", n, na, nb, 40 + n, z2, du)
    par = None
    if z2:
        mask = sum(3 << (2 * p) for p in range(n) if p % 2)
        ref = sum(1 << (2 * p) for p in range(na)) + sum(2 << (2 * p) for p in range(nb))
        par = (mask, bin(ref & mask).count("1") % 2)
    x = _dets(n, na, nb, m, n, par)
    cnt = torch.arange(1, x.numel() + 1, dtype=torch.int64, device="cuda")
    a, b = A.local_energy(model, ham, x, cnt), _static(A, model, ham, x, cnt)
    assert all(torch.equal(u, v) for u, v in zip(a, b))
    # a workspace sized for more samples, and rows counted on the device
    ws = A._ws(A.local_energy_workspace_bytes(model, ham, 4 * x.numel() + 3), "cuda")
    c = A.local_energy(model, ham, x, cnt, workspace=ws)
    assert all(torch.equal(u, v) for u, v in zip(a, c))
    nd = torch.tensor([x.numel()], dtype=torch.int64, device="cuda")
    pad = torch.cat([x, x[:1].expand(5)])
    d = A.local_energy(model, ham, pad, torch.cat([cnt, cnt[:1].expand(5)]), n_dev=nd)
    assert all(torch.allclose(u[:v.numel()], v, rtol=1e-12, atol=1e-12) for u, v in zip(d, a))


# Sectors too large for a stored prefix list whose connected determinants outnumber the determinants fourfold (every
# bit set at once, the last word of a level partly) or stay just below; the first with more samples than one CTA's statistics
# take.  The statistics: sums of about 1e3 FP64 terms in another order, each good to 1e-16 of the largest.
@pytest.mark.parametrize("kind", ["mlp", "tf"])
@pytest.mark.parametrize("n,na,nb,m", [(9, 4, 5, 1100), (10, 6, 5, 750), (11, 4, 5, 560), (11, 4, 5, 500)])
def test_calls_that_cover_the_sector(A, kind, n, na, nb, m):
    model, ham = _problem(A, kind, "fp32", n, na, nb, 70 + n)
    x = _dets(n, na, nb, m, n)
    cnt = torch.arange(1, m + 1, dtype=torch.int64, device="cuda")
    a, b = A.local_energy(model, ham, x, cnt), _static(A, model, ham, x, cnt)
    assert all(torch.equal(u, v) for u, v in zip(a, b))
    e, w = torch.complex(a[0], a[1]), cnt.double() / cnt.sum()
    mean = (w * e).sum()
    ref = torch.stack([mean.real, mean.imag, (w * (e - mean).abs() ** 2).sum(), cnt.sum().double()])
    assert torch.allclose(a[2], ref, rtol=1e-12, atol=1e-12 * float(e.abs().max()) ** 2)
    few = torch.tensor([9], dtype=torch.int64, device="cuda")  # room for many, few there: the bitmap's own bits
    c, d = A.local_energy(model, ham, x, cnt, n_dev=few), _static(A, model, ham, x[:9].contiguous(), cnt[:9])
    assert all(torch.allclose(u[:9], v, rtol=1e-12, atol=1e-12) for u, v in zip(c[:2], d))


@pytest.mark.parametrize("kind,form", [("mlp", "bf16"), ("tf", "bf16"), ("nade", "fp32")])
@pytest.mark.parametrize("n,na,nb,m", SHAPES + [(13, 6, 7, 40)])
@pytest.mark.parametrize("du", [0, 2])
def test_reuse_forms_match_amplitudes_of_the_connected_list(A, kind, form, n, na, nb, m, du):
    model, ham = _problem(A, kind, form, n, na, nb, 60 + n, du=min(du, n))
    x = _dets(n, na, nb, m, 3 * n)
    ere, eim, _ = A.local_energy(model, ham, x, torch.ones_like(x))
    if ham.n_connected == 0:  # the diagonal element alone (anqs_connected takes no empty list)
        other, _ = _problem(A, "mlp", "fp32", n, na, nb, 60 + n)
        ref = A.local_energy(other, ham, x)
        assert torch.equal(ere, ref[0]) and torch.equal(eim, ref[1])
        return
    xp, hv, _, hd = A.connected(ham, x)
    la, ph = A.logpsi(model, ham, x)
    lp, pp = (t.view(xp.shape).double() for t in A.logpsi(model, ham, xp.reshape(-1)))
    r = torch.exp(lp - la.double()[:, None])
    dp = pp - ph.double()[:, None]
    e = torch.complex(hd + (hv * r * torch.cos(dp)).sum(1), (hv * r * torch.sin(dp)).sum(1))
    bound = 1e-9 + 4e-5 * (hv.abs() * r).sum(1)
    assert torch.all((ere - e.real).abs() <= bound) and torch.all((eim - e.imag).abs() <= bound)


# sectors without a prefix index (csrc/trie.cu): few and many electrons, full shells of one spin, and pruning
@pytest.mark.parametrize("n,na,nb,m,du", [(19, 1, 1, 5, 0), (20, 2, 1, 40, 0), (21, 21, 2, 7, 1), (24, 0, 2, 3, 0),
                                          (32, 2, 30, 6, 2)])
def test_prefix_trees_match_amplitudes_of_the_connected_list(A, n, na, nb, m, du):
    test_reuse_forms_match_amplitudes_of_the_connected_list(A, "tf", "bf16", n, na, nb, m, du)


def test_prefix_trees_in_groups(A):
    """24 samples of 26 orbitals (more than one group of keys and values) against two calls of 12, bit for bit, and
    the excitations' order against anqs_connected's elements through a sum rule: for a constant amplitude E_loc is
    the row sum of the Hamiltonian."""
    from synthetic import flatten_tf, integrals, tf_params
    n, ne = 26, 9
    h, g, e = integrals(5, n, 8)
    ham = A.Hamiltonian(h, g, e, ne, ne)
    P = tf_params(5, n, 128, 4, bias_std=0.1)
    model = A.Model.transformer(n, 128, 8, 4, torch.tensor(flatten_tf(P), device="cuda"), "bf16")
    x = _dets(n, ne, ne, 24, 8)
    cnt = torch.ones_like(x)
    a = A.local_energy(model, ham, x, cnt)
    halves = [A.local_energy(model, ham, x[k:k + 12].contiguous(), cnt[:12]) for k in (0, 12)]
    for i in range(2):
        assert torch.equal(a[i], torch.cat([v[i] for v in halves]))
    P["head_w"][:] = 0  # all logits and phases equal: |psi|^2 uniform over each slot's allowed outcomes, phase zero
    P["head_b"][:] = 0
    flat = A.Model.transformer(n, 128, 8, 4, torch.tensor(flatten_tf(P), device="cuda"), "bf16")
    xp, hv, _, hd = A.connected(ham, x[:4].contiguous())
    la = A.logpsi(flat, ham, x[:4].contiguous())[0].double()
    lp = A.logpsi(flat, ham, xp.reshape(-1))[0].view(xp.shape).double()
    w = hv * torch.exp(lp - la[:, None])
    ere, eim, _ = A.local_energy(flat, ham, x[:4].contiguous())
    assert torch.all((ere - hd - w.sum(1)).abs() <= 1e-9 + 4e-5 * w.abs().sum(1)) and torch.all(eim == 0)


@pytest.mark.parametrize("kind,form,n", [("mlp", "fp32", 6), ("mlp", "bf16", 6), ("tf", "bf16", 6), ("nade", "fp32", 6),
                                         ("tf", "bf16", 20)])
def test_determinants_outside_the_sector(A, kind, form, n):
    """NaN for rows with other electron counts or bits beyond the orbitals; the other rows as without them."""
    model, ham = _problem(A, kind, form, n, 3, 2, 7)
    x = _dets(n, 3, 2, 20, 1)
    ref = A.local_energy(model, ham, x)
    high = 1 << (2 * n)
    bad = torch.cat([x[:7], torch.tensor([0, high, high | int(x[0]), -1], device="cuda"), x[7:]])
    ere, eim, _ = A.local_energy(model, ham, bad)
    assert torch.isnan(ere[7:11]).all() and torch.isnan(eim[7:11]).all()
    keep = torch.cat([torch.arange(7), torch.arange(11, bad.numel())]).cuda()
    if form == "bf16" or kind == "nade":  # in the FP32 forms a row's last bits follow its place in the list
        assert torch.allclose(ere[keep], ref[0], rtol=1e-12, atol=1e-12)
        assert torch.allclose(eim[keep], ref[1], rtol=1e-12, atol=1e-12)
    else:
        assert torch.allclose(ere[keep], ref[0], rtol=0, atol=1e-3)


def test_index_arithmetic_over_the_supported_range():
    """Division by multiplication (FastDiv) for every divisor and the values it meets."""
    for d in range(2, 513):
        m = (0xFFFFFFFF + d) // d
        v = np.unique(np.concatenate([np.arange(0, 512 * d, max(1, d // 3)), np.arange(1, 512) * d,
                                      np.arange(1, 512) * d - 1])).astype(np.uint64)
        assert np.array_equal((v * np.uint64(m)) >> np.uint64(32), v // np.uint64(d)), d
    assert math.comb(31, 2) < 512 and 16 * 16 <= 256


# Transformer adjoint over distinct prefixes: heads of width 2 and 16, one sample and a whole level, repeated samples
# (their cotangents add up), rows outside the sector (no contribution), parameters at an odd float offset, and more
# orbitals than the prefix index covers (one row per sample and position).  The same bar as the other adjoint tests.
@pytest.mark.parametrize("n,na,nb,heads,m", [(1, 1, 0, 4, 1), (3, 1, 2, 32, 1), (6, 3, 3, 4, 90), (9, 2, 7, 32, 300),
                                             (11, 5, 5, 4, 257), (20, 3, 2, 4, 40)])
def test_transformer_adjoint_rows(A, n, na, nb, heads, m):
    from oracle.anqs import TFAnsatz, log_psi
    from oracle.sector import molecular_isphys
    from synthetic import flatten_tf, integrals, tf_params
    P = tf_params(n, n, 64, 2, bias_std=0.2)
    flat = flatten_tf(P)
    params = torch.zeros(flat.size + 1, device="cuda")[1:]
    params.copy_(torch.tensor(flat))
    h, g, e = integrals(n, n, 2)
    ham = A.Hamiltonian(h, g, e, na, nb)
    model = A.Model.transformer(n, 64, heads, 2, params)
    x = _dets(n, na, nb, m, 5 * n)
    rng = np.random.default_rng(n)
    x = torch.cat([x, x[: max(1, x.numel() // 3)]])
    ca, cp = rng.normal(size=x.numel()), rng.normal(size=x.numel())
    om, ip = TFAnsatz(P, n, heads), molecular_isphys(n, na, nb)
    ps = om.parameters()
    for t in ps:
        t.requires_grad_(True)
    la, ph = log_psi(om, ip, x.cpu().numpy().astype(np.uint64))
    ref = torch.autograd.grad((torch.tensor(ca) * la).sum() + (torch.tensor(cp) * ph).sum(), ps, allow_unused=True)
    ref = np.concatenate([(torch.zeros_like(t) if r is None else r).reshape(-1).numpy() for r, t in zip(ref, ps)])
    bad = torch.tensor([0 if na + nb else 1, (1 << 2 * n) | int(x[0])], device="cuda")
    dev = lambda a: torch.tensor(np.concatenate([a, [3.0, -2.0]]), device="cuda", dtype=torch.float32)
    got = A.logpsi_vjp(model, ham, torch.cat([x, bad]), dev(ca), dev(cp)).cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)


@pytest.mark.parametrize("m", [3, 1025, 1500, 5000])
def test_static_scratch_without_excitations(A, m):
    """Full and empty shells: no connected determinants, so that the static form's arrays of them are empty; repeated
    rows, also more than one CTA's statistics take.  All energies are the diagonal element: variance zero."""
    model, ham = _problem(A, "mlp", "fp32", 3, 3, 0, 43)
    assert ham.n_connected == 0
    x = torch.full((m,), 21, dtype=torch.int64, device="cuda")
    cnt = torch.arange(1, m + 1, dtype=torch.int64, device="cuda")
    ref = A.local_energy(model, ham, x[:1])[0]
    for _ in range(20):
        ere, eim, st = _static(A, model, ham, x, cnt)
        assert torch.equal(ere, ref.expand(m)) and not eim.any()
        assert st.tolist() == [ref.item(), 0.0, 0.0, float(m * (m + 1) // 2)]


@pytest.mark.parametrize("n,value", [(6, math.nan), (6, math.inf), (20, math.nan)])
def test_transformer_adjoint_passes_nan_on(A, n, value):
    """A logit bias that is not finite makes the softmax, and so the gradient of every logit bias, NaN; the phases'
    biases keep theirs, the sum of the phase cotangents by outcome."""
    from synthetic import flatten_tf, integrals, tf_params
    P = tf_params(n, n, 64, 1, bias_std=0.2)
    P["head_b"][:] = 0
    P["head_b"][0] = value
    h, g, e = integrals(n, n, 2)
    ham = A.Hamiltonian(h, g, e, 3, 2)
    model = A.Model.transformer(n, 64, 4, 1, torch.tensor(flatten_tf(P), device="cuda"))
    x = _dets(n, 3, 2, 9, n)
    one = torch.ones(9, device="cuda")
    got = A.logpsi_vjp(model, ham, x, one, one)[-8:]
    assert torch.isnan(got[:4]).all()
    v = torch.stack([(x >> (2 * p)) & 3 for p in range(n)])
    assert torch.equal(got[4:], torch.bincount(v.flatten(), minlength=4).float())


def _reference(A, model, ham, x):
    """E_loc from anqs_connected's list and anqs_logpsi's amplitudes, and the bound of this file's docstring."""
    xp, hv, _, hd = A.connected(ham, x)
    la, ph = A.logpsi(model, ham, x)
    lp, pp = (t.view(xp.shape).double() for t in A.logpsi(model, ham, xp.reshape(-1)))
    r = torch.exp(lp - la.double()[:, None])
    dp = pp - ph.double()[:, None]
    e = torch.complex(hd + (hv * r * torch.cos(dp)).sum(1), (hv * r * torch.sin(dp)).sum(1))
    return e, 1e-9 + 4e-5 * (hv.abs() * r).sum(1)


def _launches(A, name, call):
    """What the call returns, and the timed launches of one kernel family in it."""
    from paper_2310_04166_gb300 import _lib
    lib = _lib.load()
    _lib.check(lib.anqs_profile_enable(1))
    out = call()
    torch.cuda.synchronize()
    k, ran = 0, {}
    s, c, ms = C.c_char_p(), C.c_uint64(), C.c_double()
    while lib.anqs_profile_read(k, C.byref(s), C.byref(c), C.byref(ms)) == 0:
        ran[s.value.decode()] = c.value
        k += 1
    _lib.check(lib.anqs_profile_enable(0))
    return out, ran[name]


def _agrees(A, model, ham, x, e, bound, **kw):
    ere, eim, _ = A.local_energy(model, ham, x, **kw)
    assert torch.all((ere - e.real).abs() <= bound) and torch.all((eim - e.imag).abs() <= bound)


def _tf16(A, n, na, nb, d, blocks, seed):
    from synthetic import flatten_tf, integrals, tf_params
    h, g, e = integrals(seed, n, 2 * n)
    P = tf_params(seed, n, d, blocks, bias_std=0.1)
    model = A.Model.transformer(n, d, d // 16, blocks, torch.tensor(flatten_tf(P), device="cuda"), "bf16")
    return model, A.Hamiltonian(h, g, e, na, nb)


# Enough samples (repeated where the sector has fewer) that a transformer's local energy takes the samples' prefix
# trees, one network launch per orbital: few and many electrons, full and empty shells, and a workspace that only
# holds the form over the suffixes of every connected determinant, in one launch.
@pytest.mark.parametrize("n,na,nb,m", [(19, 1, 1, 900), (20, 2, 1, 300), (21, 21, 2, 900), (24, 0, 2, 900),
                                       (32, 2, 30, 150), (32, 1, 0, 2500)])
@pytest.mark.parametrize("d", [64, 128])
def test_transformer_forms_without_an_index(A, n, na, nb, m, d):
    blocks = 2
    model, ham = _tf16(A, n, na, nb, d, blocks, 90 + n)
    x = _dets(n, na, nb, m, n)
    x = x[torch.arange(m, device="cuda") % x.numel()].contiguous()
    e, bound = _reference(A, model, ham, x)
    need = A.local_energy_workspace_bytes(model, ham, m)
    # the suffixes' scratch: 29 bytes per connected determinant, the samples' outputs, caches, keys and values
    small = m * (29 * ham.n_connected + 16 + n * (32 + 40 + 4 * blocks * d)) + 8192
    for ws, launches in ((need, n if d == 128 else None), (small, 1)):
        buf = torch.empty(ws, dtype=torch.uint8, device="cuda")
        _, ran = _launches(A, "tf_tc_amplitude_kernels", lambda: _agrees(A, model, ham, x, e, bound, workspace=buf))
        assert launches is None or ran == launches, (ws, ran)
    with pytest.raises(A.AnqsError):
        A.local_energy(model, ham, x, workspace=buf[:small // 2])
    assert model.status() == 0


@pytest.mark.parametrize("d,blocks", [(64, 1), (64, 2), (128, 2)])
@pytest.mark.parametrize("n,na,nb,m", [(6, 3, 2, 5), (10, 5, 5, 4), (10, 5, 5, 40), (12, 6, 6, 10), (18, 2, 2, 9)])
def test_transformer_forms_with_an_index(A, d, blocks, n, na, nb, m):
    """The preferred form and the suffixes of every connected determinant (few samples, or a small workspace)."""
    model, ham = _tf16(A, n, na, nb, d, blocks, 30 + n)
    x = _dets(n, na, nb, m, n + 1)
    e, bound = _reference(A, model, ham, x)
    _agrees(A, model, ham, x, e, bound)
    small = x.numel() * (29 * ham.n_connected + 16 + n * (32 + 40 + 4 * blocks * d)) + 8192
    _agrees(A, model, ham, x, e, bound, workspace=torch.empty(small, dtype=torch.uint8, device="cuda"))
    nd = torch.tensor([x.numel()], dtype=torch.int64, device="cuda")
    pad = torch.cat([x, x[:1].expand(50)])  # room for more samples than there are, in the form of more
    ere, eim, _ = A.local_energy(model, ham, pad, n_dev=nd)
    assert torch.all((ere[:x.numel()] - e.real).abs() <= bound) and torch.all((eim[:x.numel()] - e.imag).abs() <= bound)


@pytest.mark.parametrize("kind,form", [("mlp", "bf16"), ("tf", "bf16"), ("nade", "fp32"), ("mlp", "fp32"), ("tf", "fp32")])
@pytest.mark.parametrize("n,na,nb,m", [(7, 4, 3, 3), (7, 4, 3, 100), (11, 5, 4, 2), (11, 5, 4, 150), (20, 2, 1, 60)])
def test_z2_and_workspaces_of_more_samples(A, kind, form, n, na, nb, m):
    """Z2 symmetries (determinants of the other parities have no amplitude) in the forms of few and of many samples,
    with the workspace of a call of this and of twenty times as many samples."""
    model, ham = _problem(A, kind, form, n, na, nb, 40 + n, z2=True)
    mask = sum(3 << (2 * p) for p in range(n) if p % 2)
    ref = sum(1 << (2 * p) for p in range(na)) + sum(2 << (2 * p) for p in range(nb))
    x = _dets(n, na, nb, m, n, (mask, bin(ref & mask).count("1") % 2))
    e, bound = _reference(A, model, ham, x)
    for k in (1, 20):
        ws = A._ws(A.local_energy_workspace_bytes(model, ham, k * x.numel()), "cuda")
        _agrees(A, model, ham, x, e, bound, workspace=ws)


def test_batch_of_few_and_many_samples(A):
    """One persistent launch over problems by prefixes and problems by suffixes (few samples, and more orbitals than
    the index covers): as one call each, bit for bit."""
    items = []
    for n, na, nb, m in [(10, 5, 5, 3), (10, 5, 5, 300), (20, 2, 2, 12), (7, 5, 5, 200), (12, 6, 6, 2), (1, 1, 0, 1)]:
        model, ham = _problem(A, "mlp", "bf16", n, na, nb, 20 + n)
        x = _dets(n, na, nb, m, m)
        items.append(dict(model=model, ham=ham, x=x, counts=torch.arange(1, x.numel() + 1, dtype=torch.int64, device="cuda")))
    batch = A.EnergyBatch(len(items))
    for it, got in zip(items, batch.local_energy(items)):
        one = A.local_energy(it["model"], it["ham"], it["x"], it["counts"])
        assert all(torch.equal(u, v) for u, v in zip(got, one))


# The forms that sort the connected list by its first differing slot: few samples, or no prefix index.
@pytest.mark.parametrize("kind,form,n", [("mlp", "bf16", 10), ("mlp", "bf16", 20), ("nade", "fp32", 20), ("tf", "bf16", 12)])
def test_determinants_outside_the_sector_in_the_list_forms(A, kind, form, n):
    test_determinants_outside_the_sector(A, kind, form, n)


@pytest.mark.parametrize("kind,form", [("mlp", "bf16"), ("tf", "bf16"), ("nade", "fp32"), ("mlp", "fp32"), ("tf", "fp32")])
@pytest.mark.parametrize("n,na,nb,m", [(5, 5, 0, 3), (20, 20, 0, 1), (20, 20, 20, 1500)])
def test_without_excitations(A, kind, form, n, na, nb, m):
    """One determinant and no connected one: E_loc is the diagonal element, which the FP32 MLP's form also gives."""
    model, ham = _problem(A, kind, form, n, na, nb, 5)
    assert ham.n_connected == 0
    x = _dets(n, na, nb, 1, 1).expand(m).contiguous()
    other, _ = _problem(A, "mlp", "fp32", n, na, nb, 5)
    ref = A.local_energy(other, ham, x[:1])[0]
    ere, eim, st = A.local_energy(model, ham, x, torch.ones_like(x))
    assert torch.allclose(ere, ref.expand(m), rtol=1e-13) and not eim.any()
    assert torch.allclose(st, torch.tensor([ref.item(), 0.0, 0.0, m], dtype=torch.float64, device="cuda"), rtol=1e-13)


def test_transformer_leaves_in_chunks(A):
    """More determinants than one chunk of 2^20 may hold (14 orbitals, 400 samples: a bound of 1.35e6), and the same
    buffers with 30 rows, whose determinants leave the second chunk empty."""
    model, ham = _tf16(A, 14, 7, 7, 64, 1, 3)
    x = _dets(14, 7, 7, 400, 4)
    assert x.numel() * (ham.n_connected + 1) > 1 << 20
    e, bound = _reference(A, model, ham, x)
    _agrees(A, model, ham, x, e, bound)
    ere, eim, _ = A.local_energy(model, ham, x, n_dev=torch.tensor([30], dtype=torch.int64, device="cuda"))
    assert torch.all((ere[:30] - e.real[:30]).abs() <= bound[:30]) and torch.all((eim[:30] - e.imag[:30]).abs() <= bound[:30])


@pytest.mark.parametrize("kind,form", [("mlp", "bf16"), ("nade", "fp32"), ("tf", "bf16")])
@pytest.mark.parametrize("n,na,nb,m", [(11, 4, 5, 560), (11, 4, 5, 500), (9, 4, 5, 1100)])
def test_reuse_forms_that_cover_the_sector(A, kind, form, n, na, nb, m):
    """Just above and below four connected determinants per determinant of the sector, and above 32: every bit set
    without looking, or marked; then room for as many samples with nine there."""
    model, ham = _problem(A, kind, form, n, na, nb, 80 + n)
    x = _dets(n, na, nb, m, n)
    e, bound = _reference(A, model, ham, x)
    _agrees(A, model, ham, x, e, bound)
    ere, eim, _ = A.local_energy(model, ham, x, n_dev=torch.tensor([9], dtype=torch.int64, device="cuda"))
    assert torch.all((ere[:9] - e.real[:9]).abs() <= bound[:9]) and torch.all((eim[:9] - e.imag[:9]).abs() <= bound[:9])
