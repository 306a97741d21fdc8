"""Host threads with spectra of different size in the row-coupled model
kernels: the larger one needs more dynamic shared memory than a kernel gets
without asking, which no other thread's smaller spectrum may take away."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_spectra_of_several_threads():
    import torch
    import paper_2010_01371_gb300 as psps
    rng = np.random.default_rng(3)
    errors = []

    def work(ne):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(40):          # launches without a wait between them
                    psps.psps_step(states[ne], 50, history=False)
                torch.cuda.current_stream().synchronize()
        except Exception as e:
            errors.append(e)

    states = {}
    for ne in (256, 200, 199, 198):
        spec = psps.Spectrum(rng.uniform(0.005, 0.03, (ne, 4)), rng.uniform(10.0, 1000.0, (8, ne)))
        spec.set_noise(0.4, 16)
        y = torch.rand((8, 64), device="cuda") * 1000.0 + 10.0
        states[ne] = psps.State(None, spec, None, y, None)
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(ne,)) for ne in states]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
