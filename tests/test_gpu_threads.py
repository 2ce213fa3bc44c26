"""Plans used by several host threads at a time, each on its own stream: launches whose dynamic shared
memory differs (by width, by class, by set of classes) do not disturb one another."""
import threading

import numpy as np
import pytest
import torch

from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


def plan_of(classes, precision, n=2):
    rng = np.random.default_rng(3)
    Ls = (0, 1, 2, 3, 4)
    pool = W.random_primitive_pool(rng, 4, Ls=Ls)
    q = np.concatenate([W.random_class_quartets(rng, c, n, 4, Ls=Ls) for c in classes])
    return api.eri_plan_create(pool, q, precision=precision)


# the least and the most shared memory of the same kernel: widths of [ff|ff], a low and a high class
# with a g shell on their own, in sets, and from the work queue
PAIRS = {
    "widths": (([(3, 3, 3, 3)], 8, "one"), ([(3, 3, 3, 3)], 24, "one")),
    "values": (([(3, 3, 3, 3)], 0, "one"), ([(3, 3, 3, 3)], 8, "one")),
    "classes": (([(4, 0, 0, 0)], 0, "one"), ([(4, 4, 4, 4)], 0, "one")),
    "sets": (([(4, 0, 0, 0), (4, 1, 0, 0)], 16, "all"), ([(4, 4, 4, 4), (4, 4, 4, 3)], 16, "all")),
    "queue": (([(1, 0, 0, 0)], 16, "queue"), ([(4, 4, 4, 4)], 16, "queue")),
}


@pytest.mark.parametrize("pair", list(PAIRS))
def test_launches_of_several_threads(pair):
    errors, results = [], {}

    def work(i, classes, bits, form, start):
        try:
            plan = plan_of(classes, "mixed")
            s = torch.cuda.Stream()
            if bits:
                nb, sb = api.eri_output_bytes(plan, bits)
                out = (torch.zeros(nb // 4, dtype=torch.int32, device="cuda"),
                       torch.zeros(sb // 4, dtype=torch.float32, device="cuda"))
            else:
                out = (torch.zeros(api.eri_output_bytes(plan, 0)[0] // 8, dtype=torch.float64, device="cuda"),)
            torch.cuda.synchronize()

            def call():
                if form == "queue":
                    api.eri_compute_compressed_queue(plan, bits, *out, s)
                elif form == "all":
                    api.eri_compute_compressed(plan, bits, *out, s)
                elif bits:
                    api.eri_compute_compressed_class(plan, W.class_id(*classes[0]), bits, *out, s)
                else:
                    api.eri_compute_class(plan, W.class_id(*classes[0]), *out, s)

            call()
            api.eri_sync(plan, s)
            want = [o.clone() for o in out]
            torch.cuda.synchronize()
            start.wait()
            for k in range(3000):
                call()
                if k % 50 == 49:
                    api.eri_sync(plan, s)
            api.eri_sync(plan, s)
            results[i] = all(torch.equal(a, b) for a, b in zip(out, want))
        except Exception as e:  # noqa: BLE001 (reported by the test)
            errors.append(e)
            start.abort()

    start = threading.Barrier(4)
    threads = [threading.Thread(target=work, args=(i, *PAIRS[pair][i % 2], start)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert results == {i: True for i in range(4)}
