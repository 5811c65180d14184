"""Bounds priced from several host threads at once: the inner kernel's dynamic
shared memory depends on the request's strikes, and a call with few of them
must not take away what a call with many has asked for."""
import threading

import pytest

from gpu_common import torch_cuda
from paper_2206_03719_gb300 import api, workloads

pytestmark = pytest.mark.gpu


def test_bounds_with_many_and_one_strike_at_once():
    torch_cuda()
    from paper_2206_03719_gb300 import build
    build.build()
    base = workloads.SMALL_FP64.replace(n_paths=512, n_steps=2, basis="s2", greeks=(), stream=3)
    many = base.replace(strikes=[85.0 + 2.0 * k for k in range(16)])
    one = base.replace(strikes=[100.0])
    want = {}
    with api.Context(workspace_bytes=64 << 20) as ctx:
        want = {n: ctx.price_bounds(w, 8, 128) for n, w in (("many", many), ("one", one))}
    errors, done = [], threading.Event()

    def work(name, wl, calls):
        try:
            with api.Context(workspace_bytes=64 << 20) as ctx:
                for _ in range(calls):
                    if done.is_set() and name == "one":
                        break
                    got = ctx.price_bounds(wl, 8, 128)
                    assert [g["upper"] for g in got] == [g["upper"] for g in want[name]]
        except Exception as e:  # noqa: BLE001
            errors.append((name, repr(e)))
        finally:
            if name == "many":
                done.set()

    threads = [threading.Thread(target=work, args=("many", many, 600))]
    threads += [threading.Thread(target=work, args=("one", one, 100000)) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
