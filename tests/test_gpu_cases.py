"""The measured cases (perf/cases.py) call entry points that exist and work: the
smallest of each kind runs once on its own inputs."""
import random

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _finite(x):
    if isinstance(x, dict):
        return all(_finite(v) for v in x.values())
    return bool(torch.isfinite(torch.as_tensor(x)).all())


@pytest.mark.parametrize("kind", ["steps", "restart", "adjoint", "gradient", "granulation"])
def test_smallest_case_of_a_kind_runs(kind):
    from perf import cases
    rng = random.Random(1)
    pool = [c for c in cases.listed() + [cases.draw(rng) for _ in range(40)] if c["kind"] == kind]
    case = min(pool, key=lambda c: cases.work(c)["bytes"])
    out = cases.run(cases.prepare(case, 3))
    assert _finite(out)
