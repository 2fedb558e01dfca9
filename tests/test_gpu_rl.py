"""RL-stage rewards and advantages on the device (Sec. 3.4) against the
oracle, through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import cospec_rl as RL
from paper_2605_24793_gb300 import build as BLD
from paper_2605_24793_gb300 import cospec as C

from .parity_util import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    C.load_library(BLD.build())
    torch.cuda.set_device(0)
    assert C.get_device_error() == 0


def _batch(rng, groups, K, mode, max_m=6, max_r=8):
    group_off = [0]; correct = []; round_off = [0]
    match, accept, ell = [], [], []
    for x in range(groups):
        for m in range(int(rng.integers(1, max_m + 1))):
            c = {"mixed": rng.random() < 0.5, "pos": True, "neg": False}[mode]
            correct.append(int(c))
            for r in range(int(rng.integers(0, max_r + 1))):      # rollouts with no round too
                d = (rng.random(K) < 0.6).astype(np.uint8)
                a = np.where(d == 1, 1, (rng.random(K) < 0.5)).astype(np.uint8)
                match.append(d); accept.append(a)
                ell.append((-rng.exponential(1.5, K)).astype(np.float32))
            round_off.append(len(match))
        group_off.append(len(correct))
    R = len(match)
    return (np.array(group_off, np.int32), np.array(correct, np.uint8), np.array(round_off, np.int32),
            K, np.array(match, np.uint8).reshape(R, K), np.array(accept, np.uint8).reshape(R, K),
            np.array(ell, np.float32).reshape(R, K))


def _run(batch, obj=None, prm=None):
    go, co, ro, K, ma, ac, el = batch
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    kw = {}
    if obj is not None:
        kw = dict(ratio=cu(obj[0]), p_new=cu(obj[1]), p_ref=cu(obj[2]))
    out = C.rl_advantages(cu(go), cu(co), cu(ro), cu(ma), cu(ac), cu(el), prm, **kw)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


def _compare(got, ref):
    assert np.array_equal(got["eff"], ref["eff"])
    assert_close(got["g"], ref["g"], "g")
    assert np.array_equal(np.isnan(got["rho"]), np.isnan(ref["rho"]))
    assert_close(got["rho"][~np.isnan(ref["rho"])], ref["rho"][~np.isnan(ref["rho"])], "rho")
    for k in ("J", "Jbar", "adv", "adv_dec"):
        assert_close(got[k], ref[k], k)


def test_hand_case():
    go, co, ro = np.array([0, 2], np.int32), np.array([1, 0], np.uint8), np.array([0, 2, 4], np.int32)
    ma = np.array([[1, 0, 0], [1, 1, 1], [0, 1, 0], [0, 0, 1]], np.uint8)
    ac = np.array([[1, 1, 0], [1, 1, 1], [1, 1, 1], [0, 1, 1]], np.uint8)
    el = np.array([[0, -1, -3], [0, 0, 0], [-2, 0, -0.5], [-1.5, -0.7, 0]], np.float32)
    got = _run((go, co, ro, 3, ma, ac, el))
    np.testing.assert_allclose(got["J"], [1.0, -2.75], rtol=1e-6)
    np.testing.assert_allclose(got["adv"], [1.0, -1.0], rtol=1e-5)
    np.testing.assert_allclose(got["adv_dec"][2], [-2 / 2.75, 0, -0.5 / 2.75], rtol=1e-5)


@pytest.mark.parametrize("mode", ["mixed", "pos", "neg"])
@pytest.mark.parametrize("K", [6, 25, 64])
def test_matches_oracle(mode, K):
    rng = np.random.default_rng(K * 10 + {"mixed": 1, "pos": 2, "neg": 3}[mode])
    batch = _batch(rng, 60, K, mode)
    R = batch[4].shape[0]
    obj = (rng.uniform(0.5, 1.5, (R, K)).astype(np.float32),
           rng.uniform(0.05, 0.95, (R, K)).astype(np.float32),
           rng.uniform(0.05, 0.95, (R, K)).astype(np.float32))
    got = _run(batch, obj)
    ref = RL.rl_advantages(*batch, RL.RLParams(), ratio=obj[0], p_new=obj[1], p_ref=obj[2])
    _compare(got, ref)
    assert_close(got["loss"], np.array(ref["loss_terms"]), "objective terms")
    assert C.get_device_error() == 0


def test_large_batch_and_many_rounds():
    # 512 prompt groups of 8 rollouts with up to 48 rounds at K = 25
    rng = np.random.default_rng(99)
    batch = _batch(rng, 512, 25, "mixed", max_m=8, max_r=48)
    got = _run(batch)
    ref = RL.rl_advantages(*batch, RL.RLParams())
    _compare(got, ref)


def _f32_params():
    # the parameters as the library receives them
    return RL.RLParams(**{n: float(np.float32(getattr(RL.RLParams(), n)))
                          for n in ("alpha", "beta", "eta_fail", "eps", "clip_eps", "beta_h", "beta_kl")})


def _sized_batch(rng, K, sizes=(1, 0, 3, 8, 16, 17), rounds=(0, 1, 5, 33, 70)):
    """Groups of the given rollout counts (several warps per rollout, one, more rollouts than
    warps), rollouts of the given round counts."""
    correct, off = [], [0]
    for n in sizes:
        for _ in range(n):
            correct.append(int(rng.random() < 0.5))
            off.append(off[-1] + int(rng.choice(rounds)))
    R = off[-1]
    match = (rng.random((R, K)) < 0.6).astype(np.uint8)
    accept = np.where(match == 1, 1, rng.random((R, K)) < 0.7).astype(np.uint8)
    ell = (-rng.exponential(1.5, (R, K))).astype(np.float32)
    return (np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), np.array(correct, np.uint8),
            np.array(off, np.int32), K, match, accept, ell)


@pytest.mark.parametrize("policy", ["far", "near", "same", "saturated", "outside"])
@pytest.mark.parametrize("K", [1, 31, 32, 33, 64])
def test_sums_keep_their_precision(K, policy):
    """The objective's sums against 64 bits at the lane and warp boundaries.  Results are 32-bit
    roundings (6e-8); the pairs' logarithms are good to about 1e-14 absolute, the KL of two close
    policies to 1e-9 relative, the oracle's own to about 1e-7 (p / q rounded), so 1e-6 holds for
    every output."""
    rng = np.random.default_rng(K)
    batch = _sized_batch(rng, K)
    R = batch[4].shape[0]
    ratio = np.exp(0.3 * rng.standard_normal((R, K))).astype(np.float32)
    p_new = rng.uniform(0.01, 0.99, (R, K)).astype(np.float32)
    p_ref = rng.uniform(0.01, 0.99, (R, K)).astype(np.float32)
    if policy == "near":
        p_ref = (p_new * (1 + 1e-3 * rng.standard_normal((R, K)))).astype(np.float32)
    elif policy == "same":
        p_ref = p_new.copy()
    elif policy == "saturated":
        p_new[rng.random((R, K)) < 0.2] = 1.0
        p_new[rng.random((R, K)) < 0.2] = 0.0
        p_new[rng.random((R, K)) < 0.1] = 1e-9
        p_ref[rng.random((R, K)) < 0.1] = 1e-12
    elif policy == "outside":                # beyond the pairs' range: the 64-bit path
        p_new[rng.random((R, K)) < 0.3] = 1e-35
        ratio[rng.random((R, K)) < 0.2] = 1e12
        batch[6][rng.random((R, K)) < 0.2] = -1e-20
        batch[6][rng.random((R, K)) < 0.02] = -1e32
    got = _run(batch, (ratio, p_new, p_ref))
    ref = RL.rl_advantages(*batch, _f32_params(), ratio=ratio, p_new=p_new, p_ref=p_ref)
    assert np.array_equal(got["eff"], ref["eff"])
    for k in ("g", "rho", "J", "Jbar", "adv", "adv_dec"):
        scale = np.nanmax(np.abs(ref[k])) if ref[k].size else 0.0
        np.testing.assert_allclose(got[k], ref[k], rtol=1e-6, atol=1e-9 * scale, err_msg=k)
    np.testing.assert_allclose(got["loss"], np.array(ref["loss_terms"]), rtol=1e-6, atol=0 if policy != "same" else 1e-30)
    again = _run(batch, (ratio, p_new, p_ref))
    assert all(np.array_equal(got[k], again[k], equal_nan=k == "rho") for k in got)
    assert C.get_device_error() == 0


@pytest.mark.parametrize("K", [1, 3])
def test_entropy_and_kl_of_single_decisions(K):
    """One decision a call, so that nothing averages out: the result's 32-bit rounding (2^-24) and the
    pairs' error (logarithms to 3e-14, against an entropy of at least 0.03 and a KL of at least 5e-6
    here: 1e-8) are all that may show.  The relative steps from p to q lie where the KL changes from
    log(1 + r) to the difference of two logarithms (r = 2^-6) and well to both sides."""
    rng = np.random.default_rng(K)
    n = 200
    p = rng.uniform(0.05, 0.95, n).astype(np.float32)
    q = (p * (1 + rng.choice([-1, 1], n) * rng.uniform(0.01, 0.05, n))).astype(np.float32)
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device="cuda")
    match, one = torch.zeros((1, K), dtype=torch.uint8, device="cuda"), torch.ones((1, K), device="cuda")
    accept = torch.zeros((1, K), dtype=torch.uint8, device="cuda")       # the first position is rejected: one decision
    ld = np.longdouble
    for a, b in zip(p, q):
        out = C.rl_advantages(i32([0, 1]), torch.ones(1, dtype=torch.uint8, device="cuda"), i32([0, 1]), match, accept, one,
                              None, one, torch.full((1, K), float(a), device="cuda"), torch.full((1, K), float(b), device="cuda"))
        loss = out["loss"].double().cpu().numpy()
        P, Q = ld(a), ld(b)
        ent = -P * np.log(P) - (1 - P) * np.log1p(-P)
        kl = P * np.log1p((P - Q) / Q) + (1 - P) * np.log1p((Q - P) / (1 - Q))
        assert abs(loss[1] - ent) <= (2.0 ** -24 + 1e-8) * ent
        assert abs(loss[2] - kl) <= (2.0 ** -24 + 1e-8) * kl


def test_equal_returns_in_another_order_stay_equal():
    """Rollouts of the same rounds in another order have the same return.  In 64 bits a return of 64
    rounds is off by at most 9 * 2^-53 of itself (two roundings of a round's share, two in a lane's sum,
    five over the warp), which the division by sigma + eps = eps magnifies: no advantage exceeds
    2 * 9 * 2^-53 J / eps."""
    K, rounds, M = 25, 64, 8
    for seed in range(20):
        rng = np.random.default_rng(seed)
        match = (rng.random((rounds, K)) >= 0.3).astype(np.uint8)
        accept = match | (rng.random((rounds, K)) < 0.6).astype(np.uint8)
        order = np.concatenate([rng.permutation(rounds) for _ in range(M)])
        batch = (np.array([0, M], np.int32), np.ones(M, np.uint8), np.arange(0, rounds * M + 1, rounds, dtype=np.int32), K,
                 match[order], accept[order], np.zeros((rounds * M, K), np.float32))
        got = _run(batch)
        J = float(got["J"][0])
        assert np.all(got["J"] == got["J"][0])
        assert np.abs(got["adv"]).max() <= 18 * 2.0 ** -53 * J / 1e-6


@pytest.mark.parametrize("K,sizes,rounds", [
    (3, (1, 0, 2), (0, 1, 2)), (5, (4,), (1, 2, 3, 4)), (64, (1, 2), (0, 1, 33)), (7, (5, 1), (33, 70)), (31, (2, 3), (20, 33))])
def test_many_small_groups(K, sizes, rounds):
    """Both sides of the rule for small CTAs (more than 304 groups of at most 2048 decisions on average),
    groups of several tiles of 128 rounds among them."""
    rng = np.random.default_rng(K)
    batch = _sized_batch(rng, K, sizes=sizes * 160, rounds=rounds)
    R = batch[4].shape[0]
    ratio, p_new, p_ref = (rng.uniform(0.05, 0.95, (R, K)).astype(np.float32) for _ in range(3))
    got = _run(batch, (ratio, p_new, p_ref))
    ref = RL.rl_advantages(*batch, _f32_params(), ratio=ratio, p_new=p_new, p_ref=p_ref)
    assert np.array_equal(got["eff"], ref["eff"])
    for k in ("g", "rho", "J", "Jbar", "adv", "adv_dec"):
        np.testing.assert_allclose(got[k], ref[k], rtol=1e-6, atol=1e-9 * np.nanmax(np.abs(ref[k])), err_msg=k)
    np.testing.assert_allclose(got["loss"], np.array(ref["loss_terms"]), rtol=1e-6)
    assert C.get_device_error() == 0


def test_infinities_and_nan_pass_through():
    rng = np.random.default_rng(3)
    batch = _sized_batch(rng, 25)
    ell = batch[6]
    ell[rng.random(ell.shape) < 0.01] = -np.inf
    ell[rng.random(ell.shape) < 0.005] = np.nan
    got = _run(batch)
    with np.errstate(all="ignore"):
        ref = RL.rl_advantages(*batch, _f32_params())
    for k in ("g", "rho", "J", "Jbar", "adv", "adv_dec"):
        np.testing.assert_allclose(got[k], ref[k], rtol=1e-5, atol=1e-7, err_msg=k)


def test_bad_offsets_set_the_error_bit_and_skip_the_group():
    rng = np.random.default_rng(5)
    go, co, ro, K, ma, ac, el = _batch(rng, 4, 5, "mixed")
    go = go.copy()
    go[2] = go[1] - 1                                # group 1 runs backwards
    _run((go, co, ro, K, ma, ac, el))
    assert C.get_device_error() & C.DEVERR_OFFSETS
    assert C.get_device_error() == 0                 # read and cleared


def test_host_validation():
    lib = C.load_library()
    p = C.RLParams()
    fake = C.ctypes.c_void_p(1 << 20)
    args = lambda K, pr, ratio=None: (1, 1, 1, K, fake, fake, fake, fake, fake, fake,
                                      C.ctypes.byref(pr), ratio, None, None, fake, fake, fake, fake,
                                      fake, fake, fake, None, fake, 1 << 20, None)
    assert lib.cospec_rl_advantages(*args(0, p)) == -1              # K outside [1, 64]
    assert lib.cospec_rl_advantages(*args(65, p)) == -1
    assert lib.cospec_rl_advantages(*args(5, p, ratio=fake)) == -1  # objective inputs: all or none
    bad = C.RLParams(eps=0.0)
    assert lib.cospec_rl_advantages(*args(5, bad)) == -1
