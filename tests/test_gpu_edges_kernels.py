"""Kernels at the sizes where they can go wrong: edges of tiles, remainders of
chunks, the smallest and largest of their range, each against 64-bit results."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2008_11511_gb300 import build as b
    b.build()


def crandn(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def dev(x):
    return torch.tensor(np.ascontiguousarray(x), device="cuda")


# (N, frames): one frame, frames that fit one block, several chunks with a remainder
@pytest.mark.parametrize("N,frames", [(32, 1), (64, 3), (64, 700), (80, 5), (128, 513), (256, 300), (400, 53), (512, 35)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_fft2_chunks_and_remainders(N, frames, direction):
    from paper_2008_11511_gb300 import fft2
    g = torch.Generator(device="cuda").manual_seed(N + frames)
    x = torch.view_as_complex(torch.randn(frames, N, N, 2, generator=g, device="cuda"))
    f = torch.fft.fft2 if direction < 0 else torch.fft.ifft2
    ref = f(x.to(torch.complex128), norm="ortho")
    fft2(x, direction)
    per_frame = (x - ref).abs().square().sum((1, 2)).sqrt() / ref.abs().square().sum((1, 2)).sqrt()
    # 2 log2 N butterfly levels, each within a few units of 2^-24
    assert float(per_frame.max()) < 2 * np.log2(N) * 2.0 ** -24


@pytest.mark.parametrize("N,K,J", [(8, 1, 3), (12, 2, 2), (80, 1, 5), (224, 3, 3), (256, 1, 40), (400, 2, 2), (512, 1, 2)])
def test_position_shifts_at_edges(N, K, J):
    """Frames on the object's corners and edges (one-sided differences), sizes
    whose rows do not fill the last band, several modes."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N + K)
    Ho, Wo = N + 5, N + 2
    obj = (1 + 0.3 * crandn(rng, Ho, Wo)).astype(np.complex64)
    probe = crandn(rng, K, N, N)
    pos = np.stack([rng.integers(0, Ho - N + 1, J), rng.integers(0, Wo - N + 1, J)], 1).astype(np.int32)
    pos[0], pos[1] = (0, 0), (Ho - N, Wo - N)
    phi = oracle.obj_probe_to_psi(obj, probe, pos)
    psi = (phi * (1 + 0.1 * crandn(rng, *phi.shape))).astype(np.complex64)
    pb = Ptycho(dev(obj), dev(probe), torch.zeros((J, N, N), device="cuda"), pos, psi=dev(psi))
    got = pb.position_shifts(0.0).cpu().numpy()
    ref = oracle.position_shifts(obj, probe, psi, pos, 0.0)
    # the sums are of N^2 K terms of random sign and size |G| |chi|, |chi| ~ 0.1 |G| here: each term is good to
    # 2^-21, so the shift to about 2^-21 * 0.1 * sqrt(2); 1e-5 leaves room for the condition of the 2 x 2 system
    assert np.abs(got - ref).max() < 1e-5
    pb.close()


@pytest.mark.parametrize("N,K", [(12, 2), (32, 1), (64, 3), (80, 2), (128, 1), (128, 2), (256, 1), (256, 3), (400, 1),
                                 (448, 2), (512, 1), (512, 3)])
@pytest.mark.parametrize("which", ["obj", "probe", "both"])
@pytest.mark.parametrize("J", [1, 3])
def test_line_coeffs_every_form(N, K, which, J):
    """L'(0) and L''(0) over the forms of the line search (two or three waves,
    one or several modes, one frame only), with a mask, on intensities within a
    factor of the model's so that every term is well conditioned."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N + 7 * K)
    Ho, Wo = N + 4, N + 9
    obj, probe = crandn(rng, Ho, Wo), crandn(rng, K, N, N)
    d_o = 0.1 * crandn(rng, Ho, Wo) if which != "probe" else None
    d_p = 0.1 * crandn(rng, K, N, N) if which != "obj" else None
    pos = np.stack([rng.integers(0, Ho - N + 1, J), rng.integers(0, Wo - N + 1, J)], 1).astype(np.int32)

    def far(o, p):
        return np.fft.fft2(oracle.obj_probe_to_psi(o.astype(complex), p.astype(complex), pos), norm="ortho")

    A = far(obj, probe)
    B = (0 if d_p is None else far(obj, d_p)) + (0 if d_o is None else far(d_o, probe))
    C = 0 if d_o is None or d_p is None else far(d_o, d_p)
    ic = (np.abs(A) ** 2).sum(1)
    io = (ic * rng.uniform(0.3, 2.0, ic.shape)).astype(np.float32)
    mask = (rng.random((N, N)) < 0.1).astype(np.uint8)
    di = 2 * (A.conj() * B).real.sum(1)
    d2 = 2 * (np.abs(B) ** 2 + 2 * (A.conj() * C).real).sum(1)
    t1, t2 = (1 - io / ic) * di, (1 - io / ic) * d2 + io * (di / ic) ** 2
    good = mask == 0
    pb = Ptycho(dev(obj), dev(probe), dev(io), pos, mask, with_psi=False)
    assert np.all(pb.line_coeffs(None, None).cpu().numpy() == 0)
    got = pb.line_coeffs(None if d_o is None else dev(d_o.astype(np.complex64)),
                         None if d_p is None else dev(d_p.astype(np.complex64))).cpu().numpy()
    pb.close()
    # a term's relative error: the waves' transforms (2 log2 N levels of 2^-24 relative to the rms, terms scale
    # with |B| |A| and |B|^2) and a few roundings; 2^-18 of the sum of magnitudes covers both
    for g, t in zip(got, (t1, t2)):
        t = t[:, good]
        assert abs(g - t.sum()) < 2.0 ** -18 * np.abs(t).sum(), (g, t.sum(), np.abs(t).sum())


@pytest.mark.parametrize("N", [32, 64])
@pytest.mark.parametrize("J", [1, 5, 700])
@pytest.mark.parametrize("masked", [False, True])
def test_whole_frame_cycles(N, J, masked):
    """Small frames whose passes are one launch: DM from a given exit wave and
    AP against the oracle, one frame, fewer and more frames than blocks."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N + J)
    Ho, Wo = N + 23, N + 18
    obj = (1 + 0.3 * crandn(rng, Ho, Wo)).astype(np.complex64)
    probe = crandn(rng, 1, N, N)
    pos = np.stack([rng.integers(0, Ho - N + 1, J), rng.integers(0, Wo - N + 1, J)], 1).astype(np.int32)
    phi = oracle.obj_probe_to_psi(obj, probe, pos)
    psi = (phi * (1 + 0.1 * crandn(rng, *phi.shape))).astype(np.complex64)
    ic = (np.abs(np.fft.fft2(phi, norm="ortho")) ** 2).sum(1)
    io = (ic * rng.uniform(0.3, 2.0, ic.shape)).astype(np.float32)
    mask = (rng.random((N, N)) < 0.1).astype(np.uint8) if masked else None
    data = oracle.Data.make(io, pos, mask)

    def rel(a, b):
        return np.linalg.norm(a - b) / np.linalg.norm(b)

    # single precision: 4 transforms of log2 N levels and a dozen roundings, each 2^-24 of the rms; the
    # probe and object sums add J terms in FP32
    tol = 2.0 ** -24 * (8 * np.log2(N) + 12 + np.sqrt(J))
    for dm in (True, False):
        o, p = dev(obj), dev(probe)
        pb = Ptycho(o, p, dev(io), pos, mask, psi=dev(psi))
        l0 = float(pb.llk())
        llk = (pb.dm(1) if dm else pb.ap(1)).cpu().numpy()
        if dm:
            ro, rp, rpsi, rl = oracle.dm_cycle(obj, probe, psi, data)
        else:
            ro, rp, rl = oracle.ap_cycle(obj, probe, data)
        assert rel(o.cpu().numpy(), ro) < tol and rel(p.cpu().numpy(), rp) < tol
        if dm:
            assert rel(pb.psi.cpu().numpy(), rpsi) < tol
        else:  # the cycle's likelihood is that of the same model waves
            assert abs(l0 - rl) < 1e-6 * rl
        assert abs(llk[0] - rl) < 1e-6 * abs(rl)
        pb.close()


# (N, K, J, side): clusters of four and two blocks per tile, one block; fewer frames than blocks of a cluster
@pytest.mark.parametrize("N,K,J,side", [(64, 1, 3, 80), (64, 1, 150, 162), (64, 2, 100, 256), (128, 1, 90, 397),
                                        (192, 3, 1, 420), (256, 1, 12, 900)])
def test_object_gather_of_shared_tiles(N, K, J, side):
    """One AP cycle: object and probe against the oracle where a tile's frames
    are divided among the blocks of a cluster."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N + J)
    obj = (1 + 0.3 * crandn(rng, side, side)).astype(np.complex64)
    probe = crandn(rng, K, N, N)
    pos = rng.integers(0, side - N + 1, (J, 2)).astype(np.int32)
    phi = oracle.obj_probe_to_psi(obj, probe, pos)
    ic = (np.abs(np.fft.fft2(phi, norm="ortho")) ** 2).sum(1)
    io = (ic * rng.uniform(0.3, 2.0, ic.shape)).astype(np.float32)
    o, p = dev(obj), dev(probe)
    pb = Ptycho(o, p, dev(io), pos)
    llk = pb.ap(1).cpu().numpy()
    ro, rp, rl = oracle.ap_cycle(obj, probe, oracle.Data.make(io, pos, None))
    tol = 2.0 ** -24 * (8 * np.log2(N) + 12 + np.sqrt(J))  # as in test_whole_frame_cycles
    for a, b in ((o, ro), (p, rp)):
        assert np.linalg.norm(a.cpu().numpy() - b) < tol * np.linalg.norm(b)
    assert abs(llk[0] - rl) < 1e-6 * rl
    pb.close()


def _scan(N, K, J, masked, seed):
    rng = np.random.default_rng(seed)
    side = N + 37
    obj = (1 + 0.3 * crandn(rng, side, side + 6)).astype(np.complex64)
    probe = crandn(rng, K, N, N)
    pos = np.stack([rng.integers(0, side - N + 1, J), rng.integers(0, side + 6 - N + 1, J)], 1).astype(np.int32)
    phi = oracle.obj_probe_to_psi(obj, probe, pos)
    psi = (phi * (1 + 0.1 * crandn(rng, *phi.shape))).astype(np.complex64)
    ic = (np.abs(np.fft.fft2(phi, norm="ortho")) ** 2).sum(1)
    io = (ic * rng.uniform(0.3, 2.0, ic.shape)).astype(np.float32)
    mask = (rng.random((N, N)) < 0.1).astype(np.uint8) if masked else None
    return obj, probe, pos, psi, io, mask


# one frame; fewer and more frames than the backward pass has slots; several modes; parts of the update left out
@pytest.mark.parametrize("N,K,J,masked,upd_o,upd_p", [
    (160, 1, 40, True, True, True), (160, 2, 3, False, True, False), (192, 1, 1, True, True, True),
    (192, 3, 2, True, False, True), (224, 1, 31, False, True, True), (256, 1, 1, True, True, True),
    (256, 1, 3, False, False, True), (256, 1, 23, True, True, False),
    (256, 2, 2, True, True, True), (256, 3, 9, False, False, False), (384, 1, 1, False, True, True),
    (384, 2, 7, True, True, False), (400, 1, 26, True, True, True), (400, 3, 2, False, False, True),
    (448, 1, 5, True, True, True), (512, 1, 18, False, True, True), (512, 3, 2, True, True, True),
    (512, 2, 1, True, False, False)])
def test_split_passes_dm_cycle(N, K, J, masked, upd_o, upd_p):
    from paper_2008_11511_gb300 import Ptycho
    obj, probe, pos, psi, io, mask = _scan(N, K, J, masked, 10 * K + J)
    data = oracle.Data.make(io, pos, mask)
    o, p = dev(obj), dev(probe)
    pb = Ptycho(o, p, dev(io), pos, mask, psi=dev(psi))
    llk = pb.dm(1, update_obj=upd_o, update_probe=upd_p).cpu().numpy()
    ro, rp, rpsi, rl = oracle.dm_cycle(obj, probe, psi, data, update_obj=upd_o, update_probe=upd_p)
    tol = 2.0 ** -24 * (8 * np.log2(N) + 12 + np.sqrt(J))  # as in test_whole_frame_cycles
    for a, b in ((o, ro), (p, rp), (pb.psi, rpsi)):
        assert np.linalg.norm(a.cpu().numpy() - b) <= tol * np.linalg.norm(b)
    assert abs(llk[0] - rl) < 1e-6 * rl
    pb.close()


@pytest.mark.parametrize("N,K,J,masked", [(160, 1, 33, True), (192, 2, 3, False), (224, 1, 1, True),
                                          (256, 1, 1, False), (256, 1, 21, True), (256, 3, 4, True), (384, 1, 3, True),
                                          (400, 2, 9, False), (448, 1, 2, True), (512, 1, 11, True), (512, 3, 2, False)])
@pytest.mark.parametrize("parts", ["obj", "probe", "both"])
def test_split_passes_gradient(N, K, J, masked, parts):
    from paper_2008_11511_gb300 import Ptycho
    obj, probe, pos, _, io, mask = _scan(N, K, J, masked, 20 * K + J)
    pb = Ptycho(dev(obj), dev(probe), dev(io), pos, mask, with_psi=False)
    llk, go, gp = pb.ml_grad(grad_obj=parts != "probe", grad_probe=parts != "obj")
    rl, rgo, rgp = oracle.ml_grad(obj, probe, oracle.Data.make(io, pos, mask))
    # the weights 2 (1 - I_o / I_c), |.| <= 2 here, do not amplify the waves' errors
    tol = 2 * 2.0 ** -24 * (8 * np.log2(N) + 12 + np.sqrt(J))
    for a, b in ((go, rgo), (gp, rgp)):
        if a is not None:
            assert np.linalg.norm(a.cpu().numpy() - b) <= tol * np.linalg.norm(b)
    assert abs(float(llk) - rl) < 1e-6 * rl
    pb.close()


# probes that one cluster holds (one pixel per thread, four, the last size it takes) and the first one beyond
@pytest.mark.parametrize("N,K", [(8, 1), (12, 3), (32, 4), (64, 1), (64, 3), (128, 1), (80, 3), (128, 2)])
def test_probe_update_around_the_cluster_limit(N, K):
    """The probe's denominator maximum and normalisation, one launch up to 16384
    pixels, against the oracle, over several cycles of the same handle."""
    from paper_2008_11511_gb300 import Ptycho
    J = 4
    obj, probe, pos, psi, io, mask = _scan(N, K, J, True, 30 * K + N)
    data = oracle.Data.make(io, pos, mask)
    o, p = dev(obj), dev(probe)
    pb = Ptycho(o, p, dev(io), pos, mask, psi=dev(psi))
    tol = 2.0 ** -24 * (8 * np.log2(N) + 12 + np.sqrt(J))  # as in test_whole_frame_cycles
    for _ in range(3):
        before = p.cpu().numpy()
        pb.ap(1, update_obj=False)
        _, rp, _ = oracle.ap_cycle(obj, before.reshape(probe.shape), data, update_obj=False)
        assert np.linalg.norm(p.cpu().numpy() - rp) < tol * np.linalg.norm(rp)
    pb.close()


# whole frames, the unsplit and the split passes, one mode and several, the near field
BRIGHT = [(12, 1, 0.0), (64, 1, 0.0), (80, 2, 0.0), (128, 1, 0.0), (224, 1, 0.0), (256, 1, 0.0), (256, 3, 0.0), (400, 1, 0.0),
          (128, 1, 30.0), (256, 1, 90.0)]


@pytest.mark.parametrize("N,K,nf", BRIGHT)
def test_llk_of_bright_pixels_without_a_model(N, K, nf):
    """The likelihood of counts up to 1e13 where the model intensity is at its
    floor, 1e-30: I_o / I_c goes far beyond 2^126."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N)
    io = np.exp(rng.uniform(np.log(1e5), np.log(1e13), (2, N, N))).astype(np.float32)
    pb = Ptycho(dev(np.ones((N, N), np.complex64)), torch.zeros((K, N, N), dtype=torch.complex64, device="cuda"), dev(io),
                np.zeros((2, 2), np.int32), None, nearfield=nf)
    ref = oracle.llk_terms(np.zeros(io.shape), io.astype(np.float64), np.zeros((N, N), bool)).sum()
    # a term's logarithm is good to a few units of 2^-24 of its size
    assert abs(float(pb.llk()) - ref) < 2.0 ** -20 * ref
    pb.close()


@pytest.mark.parametrize("N,K", [(n, k) for n, k, nf in BRIGHT if not nf])
def test_projection_of_a_faint_wave_on_bright_pixels(N, K):
    """A wave of intensity 1e-29 everywhere takes the amplitude of 1e11 counts: a
    factor of 1e20 (a probe of one pixel, so that every value is known)."""
    from paper_2008_11511_gb300 import Ptycho
    probe = np.zeros((K, N, N), np.complex64)
    probe[K - 1, 0, 0] = N * np.sqrt(1e-29)
    io = np.full((1, N, N), 1e11, np.float32)
    pb = Ptycho(dev(np.ones((N, N), np.complex64)), dev(probe), dev(io), np.zeros((1, 2), np.int32), None)
    llk = float(pb.ap(1, update_obj=False, update_probe=False)[0])
    psi = pb.psi.cpu().numpy()[0, K - 1]
    want = N * np.sqrt(1e11)
    assert abs(psi[0, 0] - want) < 2.0 ** -20 * want
    ref = N * N * oracle.llk_terms(np.array([1e-29]), np.array([1e11]), np.zeros(1, bool))[0]
    assert abs(llk - ref) < 2.0 ** -20 * ref
    pb.close()


@pytest.mark.parametrize("N,K", [(32, 2), (64, 3), (128, 2), (256, 3), (512, 2)])
def test_line_coeffs_vanish_on_exact_intensities(N, K):
    """Several modes on intensities that equal the model's exactly: I_o / I_c is 1
    to the last bit by division, so L'(0) is 0.  Probes of one pixel each, and an
    object of small integers, make every model value exact."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N * K)
    J = 12
    obj = rng.integers(1, 8, (N + 3, N + J)).astype(np.complex64)
    probe = np.zeros((K, N, N), np.complex64)
    probe[:, 0, 0] = N * np.arange(1, K + 1)  # |P_k O|^2 / N^2 = (k o)^2 at every detector pixel
    pos = np.stack([np.zeros(J), np.arange(J)], 1).astype(np.int32)
    ic = (np.arange(1, K + 1) ** 2).sum() * np.abs(obj[0, :J]) ** 2
    io = np.broadcast_to(ic[:, None, None], (J, N, N)).astype(np.float32)
    d_o = (1 + rng.random((N + 3, N + J))).astype(np.complex64)
    pb = Ptycho(dev(obj), dev(probe), dev(io), pos, None, with_psi=False)
    l1, l2 = pb.line_coeffs(dev(d_o), None).cpu().numpy()
    pb.close()
    assert l1 == 0.0 and l2 > 0.0


# the last frame count of the unsplit passes and the first of the split ones; single batches and batches of several lanes
@pytest.mark.parametrize("N,J", [(384, 8), (384, 9), (400, 8), (400, 9), (448, 7), (448, 8), (512, 6), (512, 7), (512, 16)])
@pytest.mark.parametrize("lanes,batch", [(1, 0), (2, 0), (2, 4)])
def test_large_frames_around_the_split_limit(N, J, lanes, batch):
    """DM cycle of one mode: the choice of the passes by the number of frames, and
    the backward pass's slots for one lane, one batch and several batches."""
    from paper_2008_11511_gb300 import Ptycho
    obj, probe, pos, psi, io, mask = _scan(N, 1, J, True, N + J)
    data = oracle.Data.make(io, pos, mask)
    o, p = dev(obj), dev(probe)
    pb = Ptycho(o, p, dev(io), pos, mask, psi=dev(psi))
    pb.set_param("lanes", lanes)
    pb.set_param("batch_frames", batch)
    llk = pb.dm(1).cpu().numpy()
    ro, rp, rpsi, rl = oracle.dm_cycle(obj, probe, psi, data)
    tol = 2.0 ** -24 * (8 * np.log2(N) + 12 + np.sqrt(J))  # as in test_whole_frame_cycles
    for a, b in ((o, ro), (p, rp), (pb.psi, rpsi)):
        assert np.linalg.norm(a.cpu().numpy() - b) <= tol * np.linalg.norm(b)
    assert abs(llk[0] - rl) < 1e-6 * rl
    pb.close()


# clusters of four blocks whose tiles have from one to all of the frames; two modes; one block per tile
@pytest.mark.parametrize("N,K,J,far,side", [(64, 1, 120, 2, 300), (64, 2, 70, 1, 260), (128, 1, 150, 3, 400), (64, 1, 6, 2, 300)])
def test_object_gather_of_uneven_tiles(N, K, J, far, side):
    """Most frames on one spot and a few in the opposite corner, so that the blocks
    that share a tile outnumber its frames there: object and probe of one AP
    cycle against the oracle."""
    from paper_2008_11511_gb300 import Ptycho
    rng = np.random.default_rng(N + J)
    obj = (1 + 0.3 * crandn(rng, side, side)).astype(np.complex64)
    probe = crandn(rng, K, N, N)
    pos = rng.integers(0, 9, (J, 2)).astype(np.int32)
    pos[:far] = side - N - np.arange(far)[:, None]
    phi = oracle.obj_probe_to_psi(obj, probe, pos)
    ic = (np.abs(np.fft.fft2(phi, norm="ortho")) ** 2).sum(1)
    io = (ic * rng.uniform(0.3, 2.0, ic.shape)).astype(np.float32)
    o, p = dev(obj), dev(probe)
    pb = Ptycho(o, p, dev(io), pos)
    pb.ap(1)
    ro, rp, _ = oracle.ap_cycle(obj, probe, oracle.Data.make(io, pos, None))
    tol = 2.0 ** -24 * (8 * np.log2(N) + 12 + np.sqrt(J))  # as in test_whole_frame_cycles
    for a, b in ((o, ro), (p, rp)):
        assert np.linalg.norm(a.cpu().numpy() - b) < tol * np.linalg.norm(b)
    pb.close()


@pytest.mark.parametrize("N,K", [(256, 1), (512, 1), (512, 2)])
@pytest.mark.parametrize("form", [1, 2])
def test_tensor_core_projection_of_a_faint_wave(N, K, form):
    """test_projection_of_a_faint_wave_on_bright_pixels in the tensor-core forms."""
    from paper_2008_11511_gb300 import Ptycho
    probe = np.zeros((K, N, N), np.complex64)
    probe[K - 1, 0, 0] = N * np.sqrt(1e-29)
    io = np.full((1, N, N), 1e11, np.float32)
    pb = Ptycho(dev(np.ones((N, N), np.complex64)), dev(probe), dev(io), np.zeros((1, 2), np.int32), None)
    pb.set_param("tc", form)
    llk = float(pb.ap(1, update_obj=False, update_probe=False)[0])
    want = N * np.sqrt(1e11)
    assert abs(pb.psi.cpu().numpy()[0, K - 1, 0, 0] - want) < 1e-5 * want  # the forms' tolerance in the parity tests
    ref = N * N * oracle.llk_terms(np.array([1e-29]), np.array([1e11]), np.zeros(1, bool))[0]
    assert abs(llk - ref) < 1e-5 * ref
    pb.close()


@pytest.mark.parametrize("N", [128, 256])
@pytest.mark.parametrize("param", ["persistent", "tma"])
def test_faint_wave_in_the_other_schedules(N, param):
    """The same in the persistent schedule and the column pass fed by tensor copies."""
    from paper_2008_11511_gb300 import Ptycho
    probe = np.zeros((1, N, N), np.complex64)
    probe[0, 0, 0] = N * np.sqrt(1e-29)
    io = np.full((2, N, N), 1e11, np.float32)
    pb = Ptycho(dev(np.ones((N, N), np.complex64)), dev(probe), dev(io), np.zeros((2, 2), np.int32), None)
    pb.set_param(param, 1)
    llk = float(pb.ap(1, update_obj=False, update_probe=False)[0])
    want = N * np.sqrt(1e11)
    assert np.abs(pb.psi.cpu().numpy()[:, 0, 0, 0] - want).max() < 2.0 ** -20 * want
    ref = 2 * N * N * oracle.llk_terms(np.array([1e-29]), np.array([1e11]), np.zeros(1, bool))[0]
    assert abs(llk - ref) < 2.0 ** -20 * ref
    pb.close()
