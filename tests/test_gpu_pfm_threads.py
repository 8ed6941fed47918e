"""Two FP64 phase-field solvers of different sizes, stepped from two host threads
at once: nothing that one of them sets for its launches may reach the other's."""
import threading

import pytest

from paper_1112_5547_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_solvers_of_two_sizes_in_two_threads():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, phase_field
    build.build()

    def solver(shape, stream=None):
        a, b = inputs.drop(shape, min(shape) / 4.0, rho_hi=1.2, rho_lo=0.2, seed=9)
        return phase_field.PFM(shape, 1.4, 0.6, 0.3, 0.1, "f64", stream=stream).init(a - b)

    # rows of 512 and 1024 points: 71 and 142 KB of shared memory in the row kernel
    shapes, calls, steps = [(256, 512), (128, 1024)], 20, 400
    solvers = [solver(s, torch.cuda.Stream()) for s in shapes]
    torch.cuda.synchronize()
    errors = []

    def run(s):
        try:
            for _ in range(calls):
                s.step(steps)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(repr(e))

    threads = [threading.Thread(target=run, args=(s,)) for s in solvers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    got = [s.fields() for s in solvers]
    torch.cuda.synchronize()  # each on its solver's stream
    for shape, fields in zip(shapes, got):  # as one solver at a time gives
        for x, y in zip(fields, solver(shape).step(calls * steps).fields()):
            assert torch.equal(x, y)
