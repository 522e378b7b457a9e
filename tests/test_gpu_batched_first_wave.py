"""The phased plan whose full first waves run one problem per cluster of two blocks, asked for by its
options (the autotuner would choose it by time): every problem has the oracle's bits."""
import pytest
import torch

import oracle
import paper_2607_01735_gb300 as rb

from test_gpu_batched import _assert_bits, _batch, _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_01735_gb300 import build
    build.build_library()
    rb.load_library()


def _wave(team):
    """Clusters of two blocks that run at once: of 100 problems, one wave (51 to 100 clusters fit)."""
    _run(_batch([7] * 100, 1), 0.0, check_every=1, max_sweeps=1, team_size=team, tblock_k=2)
    assert rb.rbgs_batched_last_first_team() == 2
    return rb.rbgs_batched_last_shape()["first"]


@pytest.mark.parametrize("precision", [rb.RBGS_FP64, rb.RBGS_FP32_REFINE])
@pytest.mark.parametrize("team", [2, 4])
@pytest.mark.parametrize("over,smaller", [(0, []), (0, [15, 7]), (1, []), (4, [15, 11, 9, 7]), (-1, [15])])
def test_first_wave_by_clusters_matches_the_oracle(over, smaller, team, precision):
    """Exactly a wave of problems at the largest size, one more, a few more with smaller ones, and
    one fewer (no first phase)."""
    shape, wave = rb.rbgs_batched_last_shape, _wave(team)
    batch = _batch([23] * (wave + over) + smaller, 12)
    res, outs = _run(batch, 0.0, check_every=10, max_sweeps=20, team_size=team, tblock_k=2, precision=precision,
                     inner_sweeps=10)
    assert shape()["team"] == team and shape()["first"] == (0 if over < 0 else wave)
    assert rb.rbgs_batched_last_first_team() == (0 if over < 0 else 2)
    assert shape()["nteam"] == (wave + over if over < 0 else over)
    for (n, h2, f, u0), r, got in zip(batch, res, outs):
        ref = u0.copy()
        if precision == rb.RBGS_FP64:
            oracle.sweeps(ref, f, h2, 20)
            assert r["status"] == rb.RBGS_ENOTCONV and r["sweeps"] == 20
        else:
            oracle.refine_solve(ref, f, h2, 0.0, 10, 20)
        _assert_bits(got, ref)


def test_plain_first_wave_is_the_default_of_the_phased_plan():
    _run(_batch([7] * 300, 1), 0.0, check_every=1, max_sweeps=1, team_size=4)
    assert rb.rbgs_batched_last_first_team() == 1
