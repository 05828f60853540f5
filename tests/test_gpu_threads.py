"""Host threads that run plans of different sizes through the same kernels at once:
the shared memory a kernel may use is state of the whole process, so no thread's
launch may lower it under another's."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_two_threads_on_one_kernel(lib):
    import torch
    rows = 8
    errors, checked = [], []
    start = threading.Barrier(2)

    def work(n_t, widths, seed):
        try:
            stream = torch.cuda.Stream()
            plan = lib.Plan(96, 1250.0, 1550.0, 81.92e-6, n_t, 1e-3 * np.arange(rows), widths)
            gen = torch.Generator(device="cuda").manual_seed(seed)
            D = torch.randint(0, 255 * 96, (rows, n_t), dtype=torch.int32, device="cuda", generator=gen)
            shape = (len(widths), rows)
            outs = [(torch.zeros(shape, dtype=torch.float64, device="cuda"),
                     *(torch.zeros(shape, dtype=torch.int32, device="cuda") for _ in range(2))) for _ in range(2)]
            torch.cuda.synchronize()
            lib.sps_snr(plan, D, *outs[0], stream=stream)
            start.wait()
            for k in range(4000):
                lib.sps_snr(plan, D, *outs[1], stream=stream)
            stream.synchronize()
            checked.append(all(torch.equal(a, b) for a, b in zip(*outs)))
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)
            start.abort()

    threads = [threading.Thread(target=work, args=a) for a in ((52000, [1, 2, 4, 8], 1), (13000, [1, 2, 4, 8], 2))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert checked == [True, True]
