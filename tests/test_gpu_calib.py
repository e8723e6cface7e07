"""GPU parity of the calibration calls (Eq. 5 and R_m = H U_m^T) against the fp64 oracle.

Tolerances: the kernels take fp16 products with fp32 sums on the tensor cores, the oracle works in fp64:
weights and moments agree to 1e-4 relative (of the largest entry for the moments); the eigen solver runs in
fp64, so on the SAME matrix its eigenvalues agree to 1e-9 and its rotation to 1e-5 (fp32 output)."""
import numpy as np
import pytest
import torch

from oracle import okq_calib_oracle as CO
from paper_2609_11582_b200 import binding as B
from paper_2609_11582_b200 import workloads as WL

pytestmark = pytest.mark.gpu
D = 128


def _case(n, group=7, seed_layer=0):
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=1, n_tokens=n)
    k, v = WL.gen_kv(w, seed_layer, n_tokens=n)
    k, v = k[0, 0].contiguous(), v[0, 0].contiguous()                      # one KV head: [n, 128]
    g = torch.Generator().manual_seed(1234 + n)
    q = (torch.randn(group, n, D, generator=g) * 1.0).to(torch.float16)    # calibration queries ~ N(0, 1)
    mod = WL.modality_layout(w, n)
    signs = WL.gen_signs(w, seed_layer)
    return q, k, v, mod, signs


@pytest.mark.parametrize("n,causal", [(300, True), (1000, True), (1000, False), (64, True), (7, False)])
def test_attention_weights(n, causal):
    q, k, v, mod, signs = _case(n)
    ws = B.calib_workspace(q.shape[0], n)
    w = B.calib_attention_weights(q.cuda(), k.cuda(), ws, causal=causal).cpu().numpy().astype(np.float64)
    ref = CO.attention_weights(q.numpy().view(np.uint16), k.numpy().view(np.uint16), causal=causal)
    assert np.isfinite(w).all()
    assert np.abs(w - ref).max() <= 1e-4 * ref.max(), np.abs(w - ref).max() / ref.max()
    # every query spreads a unit of attention: sum_j alpha = 1, so sum_j w_j <= group * n, and >= group (one-hot rows count 1)
    assert q.shape[0] * 0.99 <= w.sum() <= q.shape[0] * n * 1.0001


@pytest.mark.parametrize("n", [31, 1000, 4096 + 5])
def test_moments(n):
    q, k, v, mod, signs = _case(n)
    rng = np.random.default_rng(n)
    w = (rng.random(n) ** 4 * 37.0).astype(np.float32)                      # a wide range of weights, some tiny
    ws = B.calib_workspace(7, n)
    C = B.calib_moments(v.cuda(), torch.from_numpy(w).cuda(), mod.cuda(), ws).cpu().numpy().astype(np.float64)
    ref = CO.weighted_moments(v.numpy().view(np.uint16), w.astype(np.float64), mod.numpy())
    for m in range(3):
        scale = max(np.abs(ref[m]).max(), 1e-30)
        assert np.abs(C[m] - ref[m]).max() <= 1e-4 * scale, (m, np.abs(C[m] - ref[m]).max() / scale)
        assert (C[m] == C[m].T).all()
    zero_w = B.calib_moments(v.cuda(), torch.zeros(n).cuda(), mod.cuda(), ws)
    assert not zero_w.any()


def test_rotation_matches_oracle_on_the_same_matrix():
    n = 2048
    q, k, v, mod, signs = _case(n)
    ws = B.calib_workspace(7, n)
    w = B.calib_attention_weights(q.cuda(), k.cuda(), ws)
    C = B.calib_moments(v.cuda(), w, mod.cuda(), ws)
    torch.cuda.synchronize()
    for m in range(3):
        R, lam, sweeps = B.calib_rotation(C[m].contiguous(), signs.cuda(), ws)
        R = R.cpu().numpy().astype(np.float64); lam = lam.cpu().numpy().astype(np.float64)
        assert 1 <= int(sweeps.item()) < 30
        R_ref, lam_ref = CO.rotation_from_moment(C[m].cpu().numpy().astype(np.float64), signs.numpy())
        assert np.abs(lam - lam_ref).max() <= 1e-6 * lam_ref.max()           # fp32 output of fp64 eigenvalues
        assert np.abs(R @ R.T - np.eye(D)).max() < 1e-5
        # eigenvalues of this data are well separated at the top and nearly degenerate in the noise floor, where
        # single eigenvectors are not determined: compare what is unique, the rotated moment matrix ...
        Cm = C[m].cpu().numpy().astype(np.float64)
        H = CO.hadamard_matrix(signs.numpy())
        assert np.abs(R @ Cm @ R.T - (H * lam_ref) @ H.T).max() <= 1e-5 * lam_ref.max()
        # ... and the rotation itself on the well-separated leading eigenvectors
        gap = np.abs(np.diff(lam_ref)) / lam_ref.max()
        lead = int(np.argmax(gap < 1e-3)) if (gap < 1e-3).any() else D
        assert lead >= 8
        U_gpu, U_ref = H.T @ R, H.T @ R_ref                                   # rows: eigenvectors
        assert np.abs(U_gpu[:lead] - U_ref[:lead]).max() < 1e-4
        print(f"modality {m}: {int(sweeps.item())} sweeps, {lead} separated eigenvectors compared")


def test_end_to_end_calibration_reduces_error():
    """The rotations produced on the GPU from calibration activations quantise held-out values of their own
    modality with a smaller error than the plain Hadamard rotation (the property the paper calibrates for)."""
    from oracle import okq_oracle as O
    n = 4096
    q, k, v, mod, signs = _case(n)
    ws = B.calib_workspace(7, n)
    w = B.calib_attention_weights(q.cuda(), k.cuda(), ws)
    C = B.calib_moments(v.cuda(), w, mod.cuda(), ws)
    H = CO.hadamard_matrix(signs.numpy()).astype(np.float32)
    _, _, v2, mod2, _ = _case(n, seed_layer=0)
    levels, _ = O.codebook()

    def mse(vb, R32):
        vq = O.quantize_values(vb, np.zeros(vb.shape[0], np.uint8), np.stack([R32] * 3))
        z_hat = np.asarray(levels, dtype=np.float64)[O.unpack_codes(vq["codes"])]
        rec = (z_hat @ R32.astype(np.float64)) * O.half_to_float(vq["norm"]).astype(np.float64)[:, None]
        x = vb.view(np.float16).astype(np.float64)[: rec.shape[0]]
        return float(((rec - x) ** 2).sum() / (x ** 2).sum())

    for m in range(3):
        R, _, _ = B.calib_rotation(C[m].contiguous(), signs.cuda(), ws)
        vb = np.ascontiguousarray(v2.numpy().view(np.uint16)[mod2.numpy() == m])
        e_cal, e_had = mse(vb, R.cpu().numpy()), mse(vb, H)
        print(f"modality {m}: calibrated {e_cal:.4f}  hadamard {e_had:.4f}")
        assert e_cal < e_had


def test_attention_weights_of_large_scores():
    """Scores of several hundred (log2): nearly every query attends to one key, whose weight is 2^0 / l^2 with l close to 1.  What
    is left is the rounding of sums over some hundred queries: 2^-20 of the weights' norm."""
    q, k, v, mod, signs = _case(1000)
    q = (40 * q.float()).half()
    w = B.calib_attention_weights(q.cuda(), k.cuda(), B.calib_workspace(q.shape[0], 1000)).cpu().numpy().astype(np.float64)
    ref = CO.attention_weights(q.numpy().view(np.uint16), k.numpy().view(np.uint16), causal=True)
    assert np.linalg.norm(w - ref) <= 2.0 ** -20 * np.linalg.norm(ref), np.linalg.norm(w - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("n,G,causal", [(256, 2, True), (257, 1, True), (383, 2, False), (384, 7, True), (385, 17, True), (640, 3, True),
                                        (1025, 1, False), (2047, 1, True)])
def test_attention_weights_at_the_edges_of_the_tiles(n, G, causal):
    """Around the fewest tokens of the tensor-core form (257), whole and ragged tiles of 128, ranges of steps that cut query and key
    tiles into pieces; the workspace is exactly as long as documented and nothing behind it is written.  A weight's error is that of
    sums of a few hundred fp32 numbers: 2^-20 of the weights' norm."""
    q, k, _, _, _ = _case(n, group=G)
    nb = B.lib().okq_calib_workspace_bytes(G, n)
    buf = torch.full((nb + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    w = B.calib_attention_weights(q.cuda(), k.cuda(), buf[:nb], causal=causal)
    again = B.calib_attention_weights(q.cuda(), k.cuda(), buf[:nb], causal=causal)
    assert (buf[nb:] == 0x5a).all() and (w == again).all()
    ref = CO.attention_weights(q.numpy().view(np.uint16), k.numpy().view(np.uint16), causal=causal)
    assert np.linalg.norm(w.cpu().numpy() - ref) <= 2.0 ** -20 * np.linalg.norm(ref)


@pytest.mark.parametrize("scale", [-0.05, 0.0, 0.3])
def test_attention_weights_for_any_scale(scale):
    q, k, _, _, _ = _case(300, group=2)
    w = B.calib_attention_weights(q.cuda(), k.cuda(), B.calib_workspace(2, 300), sm_scale=scale).cpu().numpy()
    ref = CO.attention_weights(q.numpy().view(np.uint16), k.numpy().view(np.uint16), sm_scale=scale)
    assert np.linalg.norm(w - ref) <= 2.0 ** -20 * np.linalg.norm(ref)


def infinite_keys(n, G):
    """Queries whose channel 5 is negative, keys 64 .. 127 infinite in it: their scores are -inf and they get no weight."""
    g = torch.Generator().manual_seed(n)
    q, k = torch.randn(G, n, D, generator=g).half(), torch.randn(n, D, generator=g).half()
    q[..., 5] = -q[..., 5].abs() - 0.01
    k[64:128, 5] = float("inf")
    return q, k


@pytest.mark.parametrize("n,causal", [(200, True), (133, False), (256, True), (257, False), (300, True), (512, True), (640, False)])
def test_attention_weights_of_infinite_keys(n, causal):
    q, k = infinite_keys(n, 3)
    w = B.calib_attention_weights(q.cuda(), k.cuda(), B.calib_workspace(3, n), causal=causal).cpu().numpy()
    ref = CO.attention_weights(q.numpy().view(np.uint16), k.numpy().view(np.uint16), causal=causal)
    assert (w[64:128] == 0).all()
    assert np.linalg.norm(w - ref) <= 2.0 ** -20 * np.linalg.norm(ref)


def test_attention_weights_wait_that_runs_out_leaves_a_mark():
    """With every block's first tile withheld the kernels return by themselves and the weights are NaN; the same call without the
    handicap gives finite weights."""
    q, k, _, _, _ = _case(1000)
    ws = B.calib_workspace(q.shape[0], 1000)
    w = B.debug_calib_timeout(q.cuda(), k.cuda(), ws, limit_clocks=20_000_000)
    torch.cuda.synchronize()                      # returns: the kernels ended by themselves
    assert w.isnan().all()
    assert B.calib_attention_weights(q.cuda(), k.cuda(), ws).isfinite().all()


def _matrices():
    rng = np.random.default_rng(11)
    had = np.array([[1.0]])
    while had.shape[0] < D:
        had = np.block([[had, had], [had, -had]])
    Q, _ = np.linalg.qr(rng.standard_normal((D, D)))
    x = rng.standard_normal((D, D))
    low = rng.standard_normal((D, 9))
    half = rng.standard_normal((64, 64))
    spectrum = np.logspace(1, -2, D)
    cluster = spectrum.copy()
    cluster[40:60] = cluster[40]
    off = np.eye(D, k=1) + np.eye(D, k=-1)
    return {"definite": x @ x.T, "indefinite": x + x.T, "low rank": low @ low.T, "low rank + identity": low @ low.T + 2 * np.eye(D),
            "zero": np.zeros((D, D)), "identity": np.eye(D), "diagonal, repeated": np.diag(rng.integers(0, 5, D).astype(float)),
            "two equal blocks": np.kron(np.eye(2), half @ half.T), "cluster": (Q * cluster) @ Q.T, "graded": (Q * np.logspace(0, -30, D)) @ Q.T,
            "tiny": x @ x.T * 1e-33, "huge": x @ x.T * 1e33, "ones": np.ones((D, D)), "pairs": np.diag(np.abs(np.arange(D) - 63.5)) + off,
            "two eigenvalues": had, "one element": np.diag([3.0] + [0.0] * (D - 1))}


@pytest.mark.parametrize("kind", list(_matrices()))
def test_rotation_of_matrices_that_are_hard_for_a_solver(kind):
    """Repeated and clustered eigenvalues (the direct solver leaves some of these to the Jacobi one), exhausted reductions, extreme
    scales.  What is unique of the result - eigenvalues, residuals, orthogonality - to a few roundings of the fp32 outputs."""
    C32 = torch.from_numpy(_matrices()[kind]).float().contiguous()
    signs = WL.gen_signs(WL.WORKLOADS["layer7b"], 0)
    ws = torch.empty(D * D * 8, dtype=torch.uint8, device="cuda")     # the documented 128 KB
    R, lam, _ = B.calib_rotation(C32.cuda(), signs.cuda(), ws)
    Cm = C32.numpy().astype(np.float64)
    Cm = 0.5 * (Cm + Cm.T)
    U = CO.hadamard_matrix(signs.numpy()).T @ R.cpu().numpy().astype(np.float64)      # rows: eigenvectors
    lam = lam.cpu().numpy().astype(np.float64)
    ref = np.linalg.eigvalsh(Cm)[::-1]
    size = max(np.abs(ref).max(), 1e-300)
    assert (np.diff(lam) <= 0).all()
    assert np.abs(lam - ref).max() <= 2.0 ** -22 * size
    assert np.abs(U @ U.T - np.eye(D)).max() <= 1e-6
    assert np.abs(U @ Cm - lam[:, None] * U).max() <= 1e-6 * size


LEFT = {"two eigenvalues", "pairs",                            # equal eigenvalues of one tridiagonal block
        "diagonal, repeated", "one element"}                   # diagonal elements below 2^-20 of the largest


@pytest.mark.parametrize("kind", list(_matrices()))
def test_direct_solver_takes_all_matrices_but_those_meant_for_the_jacobi_one(kind):
    """So that the tests of hard matrices run the solver that they are about; calibration data is all of the direct one's."""
    signs = torch.ones(D, device="cuda")
    lam = B.debug_calib_direct(torch.from_numpy(_matrices()[kind]).float().contiguous().cuda(), signs)[1]
    assert bool(lam[0].isnan()) == (kind in LEFT)
    assert kind in LEFT or lam.isfinite().all()


@pytest.mark.parametrize("n", [256, 1000, 4096])
def test_direct_solver_takes_calibration_data(n):
    q, k, v, mod, signs = _case(n)
    ws = B.calib_workspace(7, n)
    C = B.calib_moments(v.cuda(), B.calib_attention_weights(q.cuda(), k.cuda(), ws), mod.cuda(), ws)
    for m in range(3):
        assert B.debug_calib_direct(C[m].contiguous(), signs.cuda())[1].isfinite().all()


def test_weights_that_are_none_mark_the_moments_of_their_modality():
    _, _, v, mod, _ = _case(600)
    w = torch.ones(600)
    w[mod == 1] = float("nan")
    C = B.calib_moments(v.cuda(), w.cuda(), mod.cuda(), B.calib_workspace(1, 600))
    assert C[1].isnan().all() and C[0].isfinite().all() and C[2].isfinite().all()
    assert B.calib_rotation(C[1].contiguous(), torch.ones(D, device="cuda"), B.calib_workspace(1, 600))[1].isnan().all()


@pytest.mark.parametrize("decades", [0, 2, 3, 4, 5, 6])
def test_rotation_keeps_small_eigenvalues_of_graded_matrices(decades):
    """Channels whose scales differ by up to 10^6: every eigenvalue to a few roundings of fp32, relative to itself.  Reference: singular
    values of the Cholesky factor by one-sided Jacobi rotations, which are exact to fp64 for such factors."""
    from scipy.linalg import cholesky, lapack
    rng = np.random.default_rng(5)
    x = rng.standard_normal((D, 4 * D))
    scale = np.logspace(0, -decades, D)[rng.permutation(D)]
    C32 = torch.from_numpy(x @ x.T / (4 * D) * scale[:, None] * scale).float()
    C32 = (C32 + C32.T) / 2
    Cm = C32.double().numpy()
    root = np.sqrt(np.diag(Cm))
    sv, _, _, _, _, info = lapack.dgejsv((cholesky(Cm / root[:, None] / root, lower=True) * root[:, None]).T)
    assert info == 0
    ref = np.sort(sv ** 2)[::-1]
    ws = torch.empty(D * D * 8, dtype=torch.uint8, device="cuda")
    R, lam, _ = B.calib_rotation(C32.cuda(), torch.ones(D, device="cuda"), ws)
    assert (np.abs(lam.double().cpu().numpy() - ref) <= 2.0 ** -23 * ref).all()
    U = CO.hadamard_matrix(np.ones(D)).T @ R.double().cpu().numpy()
    assert np.abs(U @ U.T - np.eye(D)).max() <= 1e-6


def test_rotation_of_channels_without_values():
    """Channels that are zero have eigenvalues that are."""
    rng = np.random.default_rng(6)
    x = rng.standard_normal((D, 4 * D))
    x[1::9] = 0
    _, lam, _ = B.calib_rotation(torch.from_numpy(x @ x.T).float().cuda(), torch.ones(D, device="cuda"),
                                 torch.empty(D * D * 8, dtype=torch.uint8, device="cuda"))
    dead = len(range(1, D, 9))
    assert (lam[-dead:] == 0).all() and (lam[:-dead] > 0).all()


def test_rotations_that_overlap_may_share_a_workspace():
    """Different matrices on streams of their own with one workspace give what each gives by itself, and the workspace stays as it was."""
    signs = WL.gen_signs(WL.WORKLOADS["layer7b"], 0).cuda()
    mats = [torch.from_numpy(_matrices()[k]).float().cuda() for k in ("definite", "indefinite", "low rank", "two eigenvalues", "cluster")]
    ws = torch.full((D * D * 8,), 0x5a, dtype=torch.uint8, device="cuda")
    alone = [B.calib_rotation(C, signs, ws) for C in mats]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in mats]
    for _ in range(5):
        got = []
        for C, st in zip(mats, streams):
            with torch.cuda.stream(st):
                got.append(B.calib_rotation(C, signs, ws))
        torch.cuda.synchronize()
        assert all((x == y).all() for a, b in zip(alone, got) for x, y in zip(a, b))
    assert (ws == 0x5a).all()


def test_rotation_of_numbers_that_are_none_ends():
    signs = WL.gen_signs(WL.WORKLOADS["layer7b"], 0).cuda()
    ws = torch.empty(D * D * 8, dtype=torch.uint8, device="cuda")
    for bad in (float("nan"), float("inf")):
        C = torch.eye(D, device="cuda")
        C[3, 4] = C[4, 3] = bad
        assert B.calib_rotation(C, signs, ws)[1].isnan().all()
    R, lam, _ = B.calib_rotation(torch.eye(D, device="cuda"), signs, ws)
    assert (lam == 1).all() and R.isfinite().all()


@pytest.mark.parametrize("n,kind", [(31, "one"), (33, "alternating"), (64, "runs"), (2049, "runs"), (4133, "ids beyond two")])
def test_moments_of_tiles_with_and_without_a_modality(n, kind):
    _, _, v, mod, _ = _case(n)
    if kind == "one":
        mod = torch.full_like(mod, 2)
    elif kind == "alternating":
        mod = (torch.arange(n) % 3).to(torch.uint8)
    elif kind == "ids beyond two":
        mod = torch.where(torch.arange(n) % 700 < 350, torch.full_like(mod, 7), mod)
    w = torch.linspace(0.0, 3.0, n)
    C = B.calib_moments(v.cuda(), w.cuda(), mod.cuda(), B.calib_workspace(1, n)).cpu().numpy().astype(np.float64)
    ref = CO.weighted_moments(v.numpy().view(np.uint16), w.numpy().astype(np.float64), mod.numpy())
    for m in range(3):   # fp32 sums of n products of numbers split to 22 bits
        assert np.abs(C[m] - ref[m]).max() <= 1e-5 * max(np.abs(ref[m]).max(), 1e-30)
        assert (C[m] == C[m].T).all()
