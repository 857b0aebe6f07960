"""The bytes by which the benchmark rates the traced L_TV sweeps (no GPU)."""
import inspect

import bench


def test_sweeps_are_rated_by_what_they_touch():
    n, J, Vs, Vt = 1000, 100, 512, 300
    assert bench.launch_bytes("k_tv_inv", n, J, Vs, Vt) == 4 * Vs              # D read
    assert bench.launch_bytes("k_tv_grad", n, J, Vs, Vt) == 8 * Vs + 32 * Vt   # D, grad; both sums read and cleared
    for name in ("k_tv", "k_tv_adam", "k_query", "k_adam", "k_nn"):
        assert bench.launch_bytes(name, n, J, Vs, Vt) == bench.alg_bytes(name, n, J, Vs, Vt)
    # every rate that is printed goes through it
    assert "= alg_bytes(" not in inspect.getsource(bench)
