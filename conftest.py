"""Lattices kept alive by a caught exception's traceback are released between tests.

A test that catches an ImbError leaves its lattice in a reference cycle (exception, traceback, frame).
Collected in the middle of a later test, its release frees device memory, which waits for the GPU:
test_host_wait_is_bounded then finds the steps it queued already done.
"""
import gc


def pytest_runtest_setup(item):
    gc.collect()
