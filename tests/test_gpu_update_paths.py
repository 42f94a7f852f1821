"""The update side's paths by size and alignment: PPO losses in one launch (up to 16384 tokens)
and in two, chunks that straddle rows, the scalar form; GAE over register rows of any whole
float4 groups. Tolerances as tests/test_gpu_ppo.py and tests/test_gpu_parity.py derive them."""
import numpy as np
import pytest
import torch

from paper_2309_00754_gb300 import hydra as H
from paper_2309_00754_gb300 import synth
from tests.helpers import O, TOL_GAE, assert_rel, dev_f32, dev_i32, host_f64
from tests.test_gpu_ppo import check, make_inputs, run_kernel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,L,misalign", [
    (1, 4, False),         # one chunk
    (3, 5, False),         # every chunk straddles, a partial last chunk
    (63, 257, False),      # 16191 tokens: one launch, several chunks a thread, odd rows
    (32, 512, False),      # 16384 tokens: the largest batch of one launch
    (701, 97, False),      # two launches: straddling chunks, a partial last chunk
    (16385, 5, False),
    (33000, 3, False),     # rows shorter than a chunk: the scalar form
    (300, 400, True),      # misaligned arrays: the scalar form
    (300, 400, False),     # two launches, whole chunks
])
@pytest.mark.parametrize("whiten", [False, True])
def test_ppo_loss_by_path(S, L, misalign, whiten):
    x = make_inputs(4000 + S + L, S, L)
    check(run_kernel(*x, 0.2, whiten, misalign=misalign), *x, 0.2, whiten)
    moments = np.array([2.0 * S * L, 0.1, 3.0 * S * L])
    dm = torch.from_numpy(moments).cuda()
    got = run_kernel(*x, 0.2, whiten, moments=dm, misalign=misalign)
    assert got[2][6] == moments[0]
    rows = slice(0, min(S, 64))  # gradients of the first rows under the caller's moments
    sub = [a[rows] for a in x]
    r = np.exp(sub[0].astype(np.float64) - sub[1])
    ref = O.ppo_loss(*sub, clip_eps=0.2, whiten=whiten, moments=moments)
    amb = (np.abs(r - 1.2) <= 1e-5) | (np.abs(r - 0.8) <= 1e-5)
    g = ref["grad_logp"]
    assert np.all((np.abs(got[0][rows] - g) <= 1e-5 * np.abs(g) + 1e-6 * np.abs(g).max()) | amb)
    np.testing.assert_allclose(got[1][rows], ref["grad_values"], rtol=1e-5, atol=1e-7 * np.abs(ref["grad_values"]).max())


def test_value_loss_of_one_launch_is_near_64_bits():
    """The cluster's eight sums are added with their rounding errors. rms over 64 batches of the
    relative error: one fp32 rounding of the result alone is up to 2^-24, 2.5e-8 rms; added plainly
    the eight made it 5.8e-8."""
    err = []
    for i in range(64):
        x = make_inputs(9000 + 7 * i, 31, 400)
        _, _, stats = run_kernel(*x, 0.2, False)
        val, ret, lengths = x[4].astype(np.float64), x[3].astype(np.float64), x[5]
        d = (val - ret)[np.arange(400)[None] < lengths[:, None]]
        err.append(stats[1] / np.mean(d * d) - 1)
    assert np.sqrt(np.mean(np.square(err))) <= 4.6e-8


def test_ppo_adv_moments_of_odd_rows():
    _, _, adv, _, _, lengths = make_inputs(61, 701, 97)
    ws = torch.empty(H.ppo_workspace_size(), dtype=torch.uint8, device="cuda")
    m = torch.zeros(3, dtype=torch.float64, device="cuda")
    H.hydra_ppo_adv_moments(dev_f32(adv), dev_i32(lengths), m, ws)
    v = adv[np.arange(97)[None] < lengths[:, None]].astype(np.float64)
    n, mean, m2 = m.cpu().tolist()
    assert n == v.size and abs(mean - v.mean()) <= 1e-5 * v.std() and abs(m2 / n - v.var()) <= 2e-5 * v.var()


@pytest.mark.parametrize("S,L", [(9, 4), (5, 124), (11, 132), (17, 260), (33, 388), (40, 400), (3, 508), (5, 516), (7, 31),
                                 (6, 33), (4, 601), (2, 4097)])
def test_gae_row_lengths(S, L):
    rew, val = synth.normal_f32(3 * L, (S, L)), synth.normal_f32(3 * L + 1, (S, L))
    lengths = synth.randint(3 * L + 2, (S,), 0, L + 1)
    lengths[0] = L
    adv, ret = (torch.full((S, L), float("nan"), device="cuda") for _ in range(2))
    H.ppo_gae(dev_f32(rew), dev_f32(val), dev_i32(lengths), 0.99, 0.95, adv, ret)
    a, r = O.gae(rew.astype(np.float64), val.astype(np.float64), lengths, 0.99, 0.95)
    assert_rel(host_f64(adv), a, TOL_GAE, "advantages")
    assert_rel(host_f64(ret), r, TOL_GAE, "returns")
    dead = np.arange(L)[None] >= lengths[:, None]
    assert not host_f64(adv)[dead].any() and not host_f64(ret)[dead].any()
