"""Which kernels a call takes, without a GPU: the library's objects linked to a fake CUDA runtime
(fake_cudart.cpp) that records launches and answers the device queries as the test says."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2309_00754_gb300 import build as B
from paper_2309_00754_gb300 import hydra as H

P = 1 << 20  # a 16-byte aligned address; the fake runtime dereferences none
BIG = 1 << 40


@pytest.fixture(scope="session")
def built(tmp_path_factory):
    B.build()
    objs = [os.path.join(B.BUILD, os.path.basename(s)[:-3] + ".o") for s in B.sources()]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    so = str(tmp_path_factory.mktemp("fake") / "libhydra_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc()))), "include")
    fake = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fake_cudart.cpp")
    subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-Wl,-Bsymbolic", "-I", cuda, fake, *objs, "-o", so],
                   check=True)
    return so


class Fake:
    def __init__(self, so):
        self.lib = ctypes.CDLL(so)
        for name, (res, args) in H._SIGNATURES.items():
            f = getattr(self.lib, name)
            f.restype, f.argtypes = res, args
        self.lib.fake_launches.restype = self.lib.fake_kernels.restype = ctypes.c_char_p

    def device(self, device=0, sms=152, pairs=76, quads=36, error=0):
        self.lib.fake_device(device, sms, pairs, quads, error)

    def launches(self):
        """[(kernel, grid x, y, z, cluster, order flag)] since the last call."""
        out = [line.split() for line in self.lib.fake_launches().decode().splitlines()]
        self.lib.fake_clear()
        return [(v[0], *map(int, v[1:])) for v in out]

    def linear(self, m, k, n, streams=2, r=0):
        """Kernels of one LoRA linear of 1 to 3 streams, its lora_downs left out."""
        if streams == 3:
            rc = self.lib.hydra_lora_linear_tri(P, 2 * P, 3 * P, m, k, n, P, P, P, P, P, r, 1.0, P, P, P, 0, P, BIG, None)
        else:
            rc = self.lib.hydra_lora_linear_algo(P, 2 * P if streams == 2 else None, m, k, n, P, P, P, r, 1.0, P, P, 0,
                                                 P, BIG, 1, None)
        assert rc == 0, H.status_string(rc)
        return [v for v in self.launches() if "lora_down" not in v[0]]

    def attention(self, nseq, p, heads):
        d = 128 * heads
        assert self.lib.hydra_causal_attention(P, nseq, p, 3 * d, heads, 128, P, d, None) == 0
        (v,) = self.launches()
        return v


@pytest.fixture()
def fake(built, tmp_path):
    """A library of its own for each test: nothing cached by another one."""
    so = str(tmp_path / "lib.so")
    f = Fake(shutil.copy(built, so))
    f.device()
    return f


def _small(v):
    return "lora_gemm_small_kernel" in v[0]


def test_linear_falls_back_where_no_cluster_fits(fake):
    """A partition that holds no cluster of four CTAs (or none at all): the tile kernel serves the call."""
    assert all(_small(v) for v in fake.linear(97, 4096, 4096) + fake.linear(97, 4096, 12288))
    fake.device(device=1, quads=0)
    for (v,) in (fake.linear(97, 4096, 4096), fake.linear(97, 4096, 12288)):  # otherwise two K slices, and one
        assert _small(v) and v[4] == 2
    fake.device(device=2, pairs=0, quads=0)
    for streams in (1, 2, 3):
        for m, kernel in ((1, "dual_lora_gemm_kernel"), (128, "dual_lora_gemm_kernel"), (200, "dual_lora_gemm_2cta_kernel")):
            (v,) = fake.linear(m, 4096, 4096, streams)
            assert kernel in v[0]


def test_every_compiled_attention_form_is_taken_by_some_shape(fake):
    forms = {k for k in fake.lib.fake_kernels().decode().split() if "causal_attention" in k}
    taken = {fake.attention(nseq, p, heads)[0] for nseq in (1, 2, 3, 8, 13, 16, 20, 27, 40)
             for p in (97, 128, 300, 384, 390, 640, 700, 768, 900, 1000, 1024) for heads in (1, 5, 12, 32)}
    assert forms == taken


def test_occupancy_is_asked_once_per_device_and_a_failed_query_is_not_kept(fake):
    fake.device(error=1)
    (v,) = fake.linear(97, 4096, 12288)
    assert "dual_lora_gemm_kernel" in v[0]
    before = fake.lib.fake_cluster_queries()
    for device in range(3):
        fake.device(device=device)
        for m in range(1, 513, 8):
            for n in (520, 1032, 4096, 12288):
                for r in (0, 16):
                    assert all(_small(v) for v in fake.linear(min(m, 128), 4096, n, 2, r))
                    fake.linear(m, 4096, n, 1, r), fake.linear(m, 4096, n, 3, r)
    assert fake.lib.fake_cluster_queries() - before <= 6  # one and two K slices


def test_gemv_takes_x_as_final_only_after_a_lora_down_that_settles(fake):
    """`x_settled` of the GEMV and `settle` of the lora_down launched right before it go together; few
    rows of a short K in one wave of 4-warp CTAs are let in at once."""
    early = set()
    for m in range(1, 9):
        for k in (8, 256, 512, 520, 4096):
            for n in (8, 776, 4096, 9712, 9728, 12288, 14592, 14600, 22016):
                for shared in (True, False):
                    assert fake.lib.hydra_lora_linear(P, None if shared else 2 * P, m, k, n, P, P, P, 8, 1.0, P, P, 0, P,
                                                      BIG, None) == 0
                    down, gemv = fake.launches()
                    assert "lora_down" in down[0] and "gemv" in gemv[0] and down[5] == gemv[5]
                    if not gemv[5]:
                        early.add((m if shared else 2 * m, k, n))
    assert early == {(m, k, n) for m in range(1, 9) for k in (8, 256, 512) for n in (9728, 12288, 14592)}
    # the two calls apart: the GEMV waits
    assert fake.lib.hydra_lora_down(P, 1, 4096, P, 8, 1.0, P, None) == 0
    assert fake.lib.hydra_dual_linear(P, 2 * P, 1, 4096, 4096, P, P, P, 8, P, P, 0, 0, None) == 0
    assert [v[5] for v in fake.launches()] == [0, 0]


@pytest.mark.parametrize("whiten", [0, 1])
def test_losses_with_the_callers_moments_make_no_pass_over_the_batch_for_them(fake, whiten):
    """One thread turns them into the loss pass's coefficients, once for all its blocks."""
    assert fake.lib.hydra_ppo_loss(P, P, P, P, P, None, 1000, 400, 0.2, whiten, P, P, P, P, P, BIG, None) == 0
    first, second = fake.launches()
    assert "ppo_ext_kernel" in first[0] and first[1:4] == (1, 1, 1) and "ppo_loss_kernel" in second[0]


def test_kernel_with_its_own_order_of_sums_is_up_to_the_sizes_alone(fake):
    """Two K slices (clusters of four) add the halves of K apart: one, two and three streams all take
    them, or none does. Any other size has the tile kernel's order in either kernel."""
    halves = 0
    for m in (1, 20, 64, 128, 129, 200, 300, 384, 448, 449, 512, 513):
        for k in (8, 1024, 2048, 2560, 4096, 5120, 11008):
            for n in (8, 776, 1536, 3000, 4096, 5120, 8192, 12288, 22016):
                split = {_small(v) and v[4] == 4 for st in (1, 2, 3) for r in (0, 16) for v in fake.linear(m, k, n, st, r)}
                assert len(split) == 1
                halves += split.pop()
    assert halves > 50


def test_many_columns_take_the_tile_kernel(fake):
    """Sizes whose 128 x 256 tiles fill the chip: the few-rows kernel took up to twice the time."""
    for m, k, n, streams in ((40, 256, 65536, 1), (40, 256, 65536, 2), (97, 512, 32000, 2), (128, 1024, 22016, 1),
                             (300, 512, 14336, 2), (200, 512, 11008, 2)):
        (v,) = fake.linear(m, k, n, streams)
        assert "dual_lora_gemm" in v[0]
    for m, k, n, streams in ((97, 4096, 22016, 2), (97, 4096, 12288, 1), (300, 4096, 4096, 1), (40, 4096, 11008, 2)):
        (v,) = fake.linear(m, k, n, streams)
        assert _small(v)


def test_three_stream_estimate_counts_the_devices_multiprocessors(fake):
    """The same tiles per multiprocessor, the same choice: half the columns on half the device."""
    def choice(device, sms, n):
        fake.device(device, sms, sms // 2, 36 * sms // 152)
        (v,) = fake.linear(100, 4096, n, 3)
        return _small(v)
    for n in (4096, 6144, 8192):
        assert choice(0, 152, 2 * n) == choice(1, 76, n), n
    assert choice(1, 76, 8192) and not choice(1, 76, 6144)


def test_rmsnorm_keeps_no_more_of_a_row_than_there_is(fake):
    """The kernel by how many elements a thread keeps: a short row with the longest one's took 1.4
    times its former time."""
    keep = {}
    for d in (8, 128, 512, 520, 1024, 1032, 2048, 2056, 4096, 11008):
        assert fake.lib.hydra_rmsnorm(P, P, 5, d, 1e-6, 5, 5, 0, P, None) == 0
        ((name, *_),) = fake.launches()
        keep[d] = int(name.split("rmsnorm_kernelILi")[1].split("E")[0])
    assert keep == {8: 1, 128: 1, 512: 1, 520: 2, 1024: 2, 1032: 4, 2048: 4, 2056: 8, 4096: 8, 11008: 8}
