"""The autotuner's choice is shared by contexts that run the same stages only, and safely by threads."""
import threading

import numpy as np
import pytest

from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def first_step_launches(nx, ny, precision, **options):
    case = W.random_two_fluid(nx, ny)
    for name, value in options.items():
        setattr(case.options, name, value)
    t = ac.Tank.from_case(case, precision=precision)
    t.physical_step(case.dt, -1.0, 2)
    n = t.kernel_launches()
    t.close()
    return n


@pytest.mark.parametrize("precision,nx", [("fp64", 53), ("mixed", 59)])
def test_each_set_of_options_is_tuned_for_itself(monkeypatch, precision, nx):
    """Sizes that no other test uses: the first tank times every variant, a second one with the same options none, and
    one whose options pick other instances times them again."""
    for name in ("AC_TILE", "AC_TILE_F64"):
        monkeypatch.delenv(name, raising=False)
    first = first_step_launches(nx, 43, precision)
    assert first_step_launches(nx, 43, precision) < first
    assert first_step_launches(nx, 43, precision, limiter_k=2) == first
    # the global step: its own minimum once for the tuner and once per iteration kernel launched
    assert first_step_launches(nx, 43, precision, local_dtau=False) > first
    assert first_step_launches(nx, 43, precision, s_max=2) > first_step_launches(nx, 43, precision, s_max=2)
    assert first_step_launches(nx, 43, precision) < first


def test_threads_tune_side_by_side():
    """Contexts of their own in threads of their own, sizes in common and not: the same states as one after another."""
    sizes = [(31 + 2 * k, 21 + k) for k in range(6)]

    def run(nx, ny, precision):
        case = W.random_two_fluid(nx, ny)
        t = ac.Tank.from_case(case, precision=precision)
        t.physical_step(case.dt, -1.0, 3)
        out = t.get_state()
        t.close()
        return out

    got, errors = {}, []

    def work(k):
        try:
            for i in range(6):
                nx, ny = sizes[(i + k) % 6]
                for precision in ("fp64", "mixed"):
                    got[k, nx, ny, precision] = run(nx, ny, precision)
        except Exception as e:   # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    # the tile that a grid is tuned to is shared from then on; tiles agree to round-off
    for (_, nx, ny, precision), state in got.items():
        for a, b in zip(state, run(nx, ny, precision)):
            assert np.abs(a - b).max() <= (1e-11 if precision == "fp64" else 1e-5) * max(np.abs(b).max(), 1.0)
