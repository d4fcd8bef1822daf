"""Tables of different sizes generated by several threads at once."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_generation_from_several_threads():
    """Each thread's tables are those it gets alone, bit for bit, whatever the others ask for."""
    from paper_2110_00256_gb300 import api
    torch.zeros(1, device="cuda")
    sizes = [(4, 8), (4, 1024), (5, 300), (3, 777)]
    params = [api.table_params(qs_n_chi=n, qs_n_xi=m, bw_n_chi=n, bw_n_xi=m) for n, m in sizes]
    alone = [api.qed_tables_copy_to_host(api.qed_tables_generate(p)) for p in params]
    start, failed = threading.Barrier(len(params)), []

    def work(k):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            for _ in range(60):
                got = api.qed_tables_copy_to_host(api.qed_tables_generate(params[k], stream))
                assert all(np.array_equal(got[name], alone[k][name]) for name in got)
        except Exception as err:  # (of a thread: reported below)
            failed.append((sizes[k], err))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(params))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
