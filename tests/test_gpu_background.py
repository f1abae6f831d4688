"""Incoherent background (AP optimisation, LLK, gradient): CUDA path vs the
FP64 oracle through the C ABI, at the FP32 tolerances of test_gpu_parity."""
import numpy as np
import pytest

import oracle
from synthetic import make_scan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL1 = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2008_11511_gb300 import build as b
    b.build()


def rel(a, b):
    a = np.asarray(a)
    b = np.asarray(b)
    return float(np.linalg.norm((a - b).ravel()) / max(np.linalg.norm(b.ravel()), 1e-300))


def dev(x):
    return torch.tensor(np.ascontiguousarray(x), device="cuda")


def _problem(N, J, nearfield=0.0, seed=70):
    """A scan whose intensities carry a smooth incoherent background (Poisson
    noise), the oracle's state after one background AP cycle as the common
    warm start, and a background guess 1.5x too high."""
    s = make_scan(f"bg{N}", N=N, J=J, Ho=2 * N + 20, Wo=2 * N + 26, seed=seed, photons=1e6, step=N / 8,
                  probe_radius=N * 0.16 if not nearfield else N * 0.35, mask_fraction=0.02, noise=False,
                  nearfield=nearfield, diffuser_phase=2.0 if nearfield else 0.0,
                  phase_coef=0.0 if nearfield else None)
    yy, xx = np.mgrid[0:N, 0:N]
    b_true = 20.0 * (1.0 + 0.5 * np.cos(2 * np.pi * yy / N) * np.cos(2 * np.pi * xx / N))
    iobs = np.random.default_rng(seed + 1).poisson(s.iobs.astype(np.float64) + b_true[None]).astype(np.float32)
    iobs[:, s.mask.astype(bool)] = 0.0
    data = oracle.Data.make(iobs, s.positions, s.mask, nearfield=nearfield)
    o, p, bg, _ = oracle.ap_cycle_background(s.obj0, s.probe0, 1.5 * b_true, data)
    return s, iobs, data, o.astype(np.complex64), p.astype(np.complex64), bg.astype(np.float32)


def _ptycho(s, iobs, o, p, bg, nearfield=0.0):
    from paper_2008_11511_gb300 import Ptycho
    return Ptycho(dev(o), dev(p), dev(iobs), s.positions, s.mask, background=dev(bg), nearfield=nearfield)


@pytest.mark.parametrize("N,J,nf", [(64, 60, 0.0), (256, 24, 0.0), (128, 30, 30.0)])
def test_background_ap_cycles_with_update(N, J, nf):
    """Two AP cycles updating O, P and the background, against the oracle."""
    s, iobs, data, o0, p0, b0 = _problem(N, J, nf)
    pb = _ptycho(s, iobs, o0, p0, b0, nf)
    llk = pb.ap(2, update_background=True).cpu().numpy()
    o, p, b = o0, p0, b0
    ls = []
    for _ in range(2):
        o, p, b, l = oracle.ap_cycle_background(o, p, b, data)
        ls.append(l)
    d = oracle.object_denominator(p, s.positions, o.shape)
    ill = d > 1e-3 * d.max()
    assert rel(pb.obj.cpu().numpy()[ill], o[ill]) < 2 * TOL1
    assert rel(pb.probe.cpu().numpy(), p) < 2 * TOL1
    assert rel(pb.background.cpu().numpy(), b) < 2 * TOL1
    np.testing.assert_allclose(llk, ls, rtol=2 * TOL1)
    pb.close()


def test_background_dm_llk_and_gradient():
    """DM and the exact LLK use I_c + B (background fixed), and so does the LLK
    gradient."""
    s, iobs, data, o0, p0, b0 = _problem(64, 60)
    d = oracle.Data.make(iobs, s.positions, s.mask, background=b0)
    pb = _ptycho(s, iobs, o0, p0, b0)
    l = float(pb.llk())
    ref = oracle.llk(o0, p0, d)
    assert abs(l - ref) < 1e-5 * ref
    llk = pb.dm(2, init_psi=True).cpu().numpy()
    o, p, psi, ls = oracle.cycles("DM", o0, p0, d, 2)
    assert rel(pb.probe.cpu().numpy(), p) < 2 * TOL1
    np.testing.assert_allclose(llk, ls, rtol=2 * TOL1)
    assert rel(pb.background.cpu().numpy(), b0) == 0.0  # not updated in DM
    pb.close()
    pb = _ptycho(s, iobs, o0, p0, b0)
    _, go, gp = oracle.ml_grad(o0, p0, d)
    _, g_o, g_p = pb.ml_grad()
    assert rel(g_o.cpu().numpy(), go) < 1e-4 and rel(g_p.cpu().numpy(), gp) < 1e-4
    pb.close()


# every column pass that updates a background: without and with the split column
# transform, M a multiple of 4 and not, one mode and several, the near field's
FORMS = [(64, 1, 0.0), (80, 2, 0.0), (128, 1, 0.0), (256, 1, 0.0), (400, 1, 0.0), (224, 2, 0.0), (512, 2, 0.0)]


def _background_only(io, bg, probe, nearfield=0.0):
    """One cycle of one frame that updates the background alone: B <- B I_o / (I_c + B)."""
    from paper_2008_11511_gb300 import Ptycho
    N = io.shape[-1]
    obj = np.ones((N, N), dtype=np.complex64)
    pb = Ptycho(dev(obj), dev(probe), dev(io[None]), np.zeros((1, 2), np.int32), None, background=dev(bg),
                nearfield=nearfield)
    pb.ap(1, update_obj=False, update_probe=False, update_background=True)
    out = pb.background.cpu().numpy()
    pb.close()
    return out


@pytest.mark.parametrize("N,K,nf", FORMS + [(128, 1, 30.0), (256, 1, 90.0)])
def test_background_quotient_over_its_range(N, K, nf):
    """No probe, so I_c = 0 and the updated background is B fl(I_o / B): I_o to
    a unit in the last place of the quotient and the rounding of the product,
    from the floor of I_c up to the largest values."""
    rng = np.random.default_rng(N + K)
    bg = np.exp(rng.uniform(np.log(1e-30), np.log(3e38), (N, N))).astype(np.float32)
    bg[0, :8] = [1e-30, 1.1e-30, 1.0, 2.0 ** 126, 2.0 ** 127, 3e38, 1e38, 3.0]
    io = (bg * np.exp(rng.uniform(np.log(1e-6), 0.0, (N, N)))).astype(np.float32)
    io[1, :4] = [0.0, -3.0, 0.0, 0.0]
    got = _background_only(io, bg, np.zeros((K, N, N), np.complex64), nf)
    want = np.maximum(io, 0.0).astype(np.float64)
    assert np.all(np.isfinite(got))
    normal = want >= 2.0 ** -126
    assert np.all(np.abs(got - want)[normal] <= 2.0 ** -22 * want[normal])
    assert np.all(got[~normal] <= 2.0 ** -126)


@pytest.mark.parametrize("N,K,nf", FORMS)
def test_background_under_an_infinite_model_intensity(N, K, nf):
    """A model intensity beyond the range of single precision leaves no
    background (I_o / inf = 0), as the exact division gives it."""
    probe = np.zeros((K, N, N), np.complex64)
    probe[0, 0, 0] = 3.2e19  # |.|^2 is infinite at every detector pixel
    io = np.full((N, N), 7.0, np.float32)
    got = _background_only(io, np.full((N, N), 5.0, np.float32), probe)
    assert np.all(got == 0.0)


# remainders of M by four (160, 224, 400), several modes, the near field with and without split passes, few large
# frames (unsplit) and more (split); odd frame counts in one batch, and in batches of 5 (dependent launches)
@pytest.mark.parametrize("N,K,J,nf", [(64, 2, 9, 0.0), (80, 1, 21, 0.0), (128, 2, 7, 0.0), (160, 1, 23, 0.0), (160, 2, 11, 0.0),
                                      (224, 1, 11, 0.0), (256, 1, 13, 0.0), (256, 2, 7, 0.0), (400, 1, 7, 0.0),
                                      (400, 1, 11, 0.0), (400, 2, 5, 0.0), (512, 1, 9, 0.0), (512, 2, 3, 0.0),
                                      (128, 1, 9, 40.0), (256, 1, 13, 90.0)])
@pytest.mark.parametrize("batch", [0, 5])
def test_background_update_in_every_pass(N, K, J, nf, batch):
    """One AP cycle that updates object, probe and background, with a mask,
    against the oracle."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N + 10 * K + J)

    def crandn(*shape):
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)

    Ho, Wo = N + 21, N + 18
    obj, probe = (1 + 0.3 * crandn(Ho, Wo)).astype(np.complex64), crandn(K, N, N)
    pos = np.stack([rng.integers(0, Ho - N + 1, J), rng.integers(0, Wo - N + 1, J)], 1).astype(np.int32)
    mask = (rng.random((N, N)) < 0.1).astype(np.uint8)
    empty = oracle.Data.make(np.zeros((J, N, N), np.float32), pos, mask, nearfield=nf)
    ic = (np.abs(empty.to_detector(oracle.obj_probe_to_psi(obj, probe, pos))) ** 2).sum(1)
    bg = (ic.mean() * rng.uniform(0.5, 1.5, (N, N))).astype(np.float32)
    io = ((ic + bg) * rng.uniform(0.3, 2.0, ic.shape)).astype(np.float32)
    io[:, mask.astype(bool)] = 0.0
    pb = Ptycho(dev(obj), dev(probe), dev(io), pos, mask, background=dev(bg), nearfield=nf)
    pb.set_param("batch_frames", batch)
    llk = pb.ap(1, update_background=True).cpu().numpy()
    ro, rp, rb, rl = oracle.ap_cycle_background(obj, probe, bg, oracle.Data.make(io, pos, mask, nearfield=nf))
    # single precision: 4 transforms (near field 8) of log2 N levels and a dozen roundings, each 2^-24 of the rms;
    # the sums add J terms in FP32.  The background is the mean of J quotients of wave intensities, twice the waves'
    # relative errors
    tol = 2.0 ** -24 * ((16 if nf else 8) * np.log2(N) + 12 + np.sqrt(J))
    assert rel(pb.obj.cpu().numpy(), ro) < tol and rel(pb.probe.cpu().numpy(), rp) < tol
    assert rel(pb.background.cpu().numpy(), rb) < 2 * tol
    assert abs(llk[0] - rl) < 1e-6 * abs(rl)
    assert np.array_equal(pb.background.cpu().numpy()[mask.astype(bool)], bg[mask.astype(bool)])
    pb.close()


@pytest.mark.parametrize("N,K,nf", FORMS + [(128, 1, 30.0), (256, 1, 90.0)])
def test_background_is_added_once_beside_bright_pixels(N, K, nf):
    """Some pixels so bright over their model (1e9 counts, 1e-29) that their
    neighbours' likelihood is computed again: the background's sums are not."""
    rng = np.random.default_rng(N + K)
    bg = rng.uniform(1.0, 100.0, (N, N)).astype(np.float32)
    io = rng.uniform(1.0, 100.0, (N, N)).astype(np.float32)
    y, x = rng.integers(0, N, (2, 9))
    bg[y, x], io[y, x] = 1e-29, 1e9
    got = _background_only(io, bg, np.zeros((K, N, N), np.complex64), nf)
    # a unit in the last place of the quotient and the rounding of the product
    assert np.abs(got.astype(np.float64) / io - 1).max() <= 2.0 ** -22
