"""Datasets created by several threads of one context at once: each call judges its own inputs."""
import threading

import numpy as np
import pytest

from paper_1511_02186_gb300 import aidw

pytestmark = pytest.mark.gpu


def test_threads_creating_datasets_judge_their_own_inputs():
    rng = np.random.default_rng(3)
    n, rounds, threads = 3001, 25, 8
    good = [rng.uniform(0.0, 10.0, n) for _ in range(3)]
    bad = [good[0], good[1], good[2].copy()]
    bad[2][n - 1] = np.nan
    wrong = []

    with aidw.Context(0) as c:
        def work(t):
            for _ in range(rounds):
                refused = False
                try:
                    ds = c.create_dataset(*(bad if t % 2 else good), 100.0)
                    ds.destroy()
                except aidw.AidwError as e:
                    refused = e.status == aidw.ERR_INVALID_ARG
                if refused != bool(t % 2):
                    wrong.append(t)

        ts = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not wrong
        assert c.check_device_errors() == aidw.OK
