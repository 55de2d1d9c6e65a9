"""Suite-wide set-up that every test file shares.

Tests that ask the driver how much device memory is free (the 1280^3 runs ask
for up to 240 GB of it) see as used what torch's caching allocator still holds
of earlier tests' tensors.  Each GPU test therefore starts with that cache
given back.
"""
import gc
import sys

import pytest


@pytest.fixture(autouse=True)
def torch_cache_given_back(request):
    torch = sys.modules.get("torch")
    if torch is not None and request.node.get_closest_marker("gpu") and torch.cuda.is_initialized():
        gc.collect()  # tensors of a finished test may sit in reference cycles
        torch.cuda.empty_cache()
    yield
