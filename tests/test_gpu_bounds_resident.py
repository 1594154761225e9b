"""The on-chip steps in the bounds-checked debug build (test_gpu_bounds.py):
every access to the state and to the exchange words is checked against its
buffer.  Single lattices and batches, periodic and walled, from one tile to
tiles of more than 256 nodes with odd sides, odd and even numbers of steps.
That the on-chip steps ran shows in the allocation of their exchange words.  A
negative control tells the checks of a shorter density buffer than there is."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SIZES = [(5, 5, False), (9, 9, True), (70, 21, False), (131, 37, True), (250, 120, False),
         (331, 173, False), (331, 173, True), (500, 201, True)]
PRECISIONS = ["f64", "f32", "f32_offset"]


def _child():
    from paper_1611_00907_gb300 import (Batch, LbmError, Simulation, _lib, eos_coexistence,
                                        inputs)
    assert os.path.basename(_lib.LIB_PATH) == "libcplbm_checked.so"
    lib = _lib.load()
    rv, rl, mc = eos_coexistence("cs", 1.0, 4.0, 1.0, 0.85)

    def field(nx, ny, walls):
        r = max(2.0, min(nx, ny) / 4)
        return (inputs.wall_drop if walls else inputs.drop)(nx, ny, r, rl, rv, 4.0)

    def held():
        return lib.lbm_test_device_allocs()

    runs = 0
    for prec in PRECISIONS:
        spec = [dict(nx=nx, ny=ny, walls=w, rho_ref=0.15, mu_bottom=mc + 0.01)
                for nx, ny, w in SIZES]
        for s in spec:
            rho = field(s["nx"], s["ny"], s["walls"])
            with Simulation(precision=prec, **s) as sim:
                sim.init(rho)
                if prec != "f64" and not s["walls"]:
                    sim.autotune()             # the default of these: tile kernels
                sim.moments()
                had = held()
                sim.step(5).moments()
                sim.step(30).moments()
                if prec == "f64" or s["walls"]:
                    assert held() == had + 1, s
                sim.reduce()
                sim.populations()
            runs += 1
        for group in (spec[2:5], spec[5:7]):
            with Batch(group, precision=prec) as b:
                for k, s in enumerate(group):
                    b.init(k, field(s["nx"], s["ny"], s["walls"]))
                b.moments(0)
                had = held()
                b.step(30)
                assert held() == had + 2
                b.step(5).step(5)
                b.set_active(1, False).step(30)
                for k in range(len(group)):
                    b.moments(k)
            runs += 1
    with Simulation(131, 70, precision="f64") as s:
        s.init(field(131, 70, False))
        assert lib.lbm_test_shrink_bounds(s._ctx, 1000) == _lib.LBM_OK
        s.step(8)
        try:
            s.moments()
            caught = False
        except LbmError as err:
            caught = "outside its buffer" in str(err)
    print(json.dumps({"runs": runs, "negative_control_caught": caught}))


@pytest.mark.gpu
def test_no_access_of_the_on_chip_steps_leaves_its_buffer():
    subprocess.run([sys.executable, "-m", "paper_1611_00907_gb300._build", "--checked"],
                   cwd=ROOT, check=True, timeout=1800)
    env = dict(os.environ, CPLBM_LIBRARY_VARIANT="checked",
               PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    res = subprocess.run([sys.executable, os.path.abspath(__file__), "child"], cwd=ROOT,
                         env=env, capture_output=True, text=True, timeout=1800)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-4000:]
    out = json.loads(res.stdout.strip().splitlines()[-1])
    assert out["runs"] == len(PRECISIONS) * (len(SIZES) + 2)
    assert out["negative_control_caught"]


if __name__ == "__main__" and sys.argv[1:] == ["child"]:
    _child()
