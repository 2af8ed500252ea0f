"""Failure detection on the GPU without a fault: a bounded wait on a barrier
that nothing completes gives up within its limit, the time-out reaches the
host as GKO_TIMEOUT through the device error word, and the context keeps
working (an SpMV afterwards matches the oracle)."""
import time

import numpy as np
import pytest

from gpu_util import check_spmv_f64, dev, host
from paper_2006_14290_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_bounded_wait_times_out_and_context_survives(gko):
    G = gko
    G.gko_device_status()  # clean start
    t0 = time.perf_counter()
    assert G.gko_diag_bounded_wait(20_000_000)  # about 10 ms at 2 GHz
    assert time.perf_counter() - t0 < 5.0
    with pytest.raises(G.GkoError) as e:
        G.gko_device_status()
    assert e.value.status == G.TIMEOUT
    G.gko_device_status()  # the word was cleared by the read
    A = I.stencil3d_27pt(12)
    M = G.from_csr(A)
    x = np.random.default_rng(0).uniform(-1, 1, A.n_cols)
    yd = dev(np.zeros(A.n_rows))
    G.gko_spmv(1.0, M, dev(x), 0.0, yd)
    check_spmv_f64(host(yd), A, x, 1.0, 0.0, None)
    G.gko_device_status()


def test_bounded_wait_rejects_bad_limits(gko):
    G = gko
    for bad in (0, -5, 2**33):
        with pytest.raises(G.GkoError) as e:
            G.gko_diag_bounded_wait(bad)
        assert e.value.status == G.INVALID_ARG


@pytest.mark.parametrize("cluster,blocks", [(1, 2), (1, 7), (1, 16), (0, 2), (0, 33), (0, 152)])
@pytest.mark.parametrize("values", [0, 1, 2, 3])
def test_exchange_totals_and_slot_words(gko, cluster, blocks, values):
    """The single-launch solvers' exchanges: every total and every published
    entry is right over more steps than the 16-bit tags count, and no word of
    a slot keeps the tag of an older step."""
    G = gko
    steps = 66_000 if blocks in (7, 33) else 500
    out, cycles = G.gko_diag_exchange(bool(cluster), blocks, values, steps)
    assert np.all(out == [steps, 0, 0, 0]), out
    assert cycles > 0
    G.gko_device_status()


def test_exchange_check_rejects_bad_sizes(gko):
    G = gko
    for bad in ((True, 1, 1, 5), (True, 17, 1, 5), (False, 161, 1, 5), (True, 4, 4, 5), (True, 4, 1, 0)):
        with pytest.raises(G.GkoError) as e:
            G.gko_diag_exchange(*bad)
        assert e.value.status == G.INVALID_ARG


@pytest.mark.parametrize("cluster,blocks", [(True, 2), (True, 7), (True, 16), (False, 2), (False, 33)])
@pytest.mark.parametrize("values", [0, 1, 3])
@pytest.mark.parametrize("leave_step", [0, 5, 49])
def test_exchange_ends_when_a_block_leaves(gko, cluster, blocks, values, leave_step):
    """A block leaves in the middle (its peers may be in a barrier, and in a
    cluster may read its shared memory later): the others' waits run out, all
    blocks end, the time-out is recorded and the context keeps working."""
    G = gko
    G.gko_device_status()
    out, _ = G.gko_diag_exchange(cluster, blocks, values, 50, blocks // 2, leave_step, 2_000_000)  # 1 ms
    assert out[blocks // 2, 0] == leave_step and np.all(out[:, 3] == 1), out
    assert np.all(out[:, 0] >= leave_step) and np.all(out[:, 0] <= 50), out
    if values:
        assert np.all(out[:, 0] == leave_step), out
    with pytest.raises(G.GkoError) as e:
        G.gko_device_status()
    assert e.value.status == G.TIMEOUT
    out, _ = G.gko_diag_exchange(cluster, blocks, values, 50)
    assert np.all(out == [50, 0, 0, 0]), out
    G.gko_device_status()
