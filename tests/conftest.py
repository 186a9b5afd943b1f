import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (run with -m gpu on a B200)")


def pytest_collection_modifyitems(config, items):
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except Exception:
        has_gpu = False
    if has_gpu:
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


@pytest.fixture(scope="session")
def known_route():
    """(permutations, the oracle's bits) of the larger inputs that several tests share, each computed once."""
    import numpy as np
    import oracle
    from paper_1912_04050_b200 import inputs
    cache = {}

    def get(kind, n, batch=1):
        if (kind, n, batch) not in cache:
            perm = (inputs.random_perm_batch(n, batch, seed0=37 * n + batch) if kind == "random"
                    else np.tile(inputs.structured_perms(n)[kind], (batch, 1)))
            cache[kind, n, batch] = perm, oracle.route(perm, n)
        return cache[kind, n, batch]

    return get
