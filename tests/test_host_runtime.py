"""The host runtime (qfs_api.cu) over a fake device: what a call allocates and launches, without a GPU.

tests/host_runtime.cu compiles the runtime with counting stand-ins for the CUDA calls and recorders for the kernel
launchers, and prints one JSON line per scenario.
"""
import json
import os
import re
import subprocess

import pytest

from test_layout_host import CSRC, ROOT, _nvcc

MB = 1 << 20
CONTROL_BYTES = 1024   # the control block and the rounding of small buffers


@pytest.fixture(scope="module")
def runtime(tmp_path_factory):
    nvcc = _nvcc()
    if not nvcc:
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("runtime") / "host_runtime")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "host_runtime.cu"), "-o", exe],
                   check=True, capture_output=True)

    def run(**kw):
        arg = ",".join(f"{k}={v}" for k, v in kw.items())
        out = subprocess.run([exe, arg], check=True, capture_output=True, text=True).stdout
        r = json.loads(out)
        r["fused"] = [{k: int(v) for k, v in re.findall(r"(\w+)=(\d+)", x)} for x in r["launches"]
                      if x.startswith("fused")]
        return r
    return run


@pytest.mark.parametrize("p,power,n,budget", [(7, 1, 1, 8 * MB), (7, 1, 2, 8 * MB), (7, 1, 600, 8 * MB),
                                              (7, 1, 100000, 1024 * MB), (7, 1, 100, 550 * MB), (5, 0, 4, 4 * MB),
                                              (5, 0, 1000, 200 * MB), (3, 0, 2, 1 * MB), (3, 1, 500, 6 * MB)])
@pytest.mark.parametrize("form", [0, 1, 2])
def test_workspace_stays_within_the_budget(runtime, p, power, n, budget, form):
    # everything but the list of screened rows (8 bytes each) counts: chain buffers and theta's classes
    r = runtime(op="heights", p1=p, n1=n, power=power, budget=budget, form=form)
    assert r["rc"] == 0 and len(r["fused"]) == 1
    assert r["peak"] <= budget + 8 * n + CONTROL_BYTES


@pytest.mark.parametrize("p,power", [(3, 0), (5, 0), (3, 1), (5, 1), (7, 1)])
def test_default_budget_takes_theta_by_rows(runtime, p, power):
    assert runtime(op="heights", p1=p, n1=100000, power=power)["fused"][0]["classes"] == 1


@pytest.mark.parametrize("p", [3, 5, 7])
def test_reduced_kernel_takes_no_workspace(runtime, p):
    # its forms live in shared memory: neither chain buffers nor classes, and no budget is too small
    for budget in (0, 1):
        r = runtime(op="heights", p1=p, n1=100000, p2=p, n2=7, power=2, budget=budget)
        assert r["rc"] == 0 and r["launches"] == ["screen", "reduced"]
        assert r["peak"] <= 8 * 100007 + CONTROL_BYTES
    # the fused kernel's reduced mode needs a quartic's buffers
    for kw in (dict(max_ctas=3), dict(p2=11, n2=1), dict(form=0)):
        r = runtime(op="heights", p1=p, n1=1000, power=2, **kw)
        assert r["rc"] == 0 and len(r["fused"]) == 1
        assert runtime(op="heights", p1=p, n1=1000, power=2, budget=1, **kw)["rc"] == 5


@pytest.mark.parametrize("groups,crew,joint", [
    (((11, 0), (5, 13000)), 8, 0),              # the one p = 11 row had height 1: every quartic by single CTAs
    (((11, 1), (5, 13000)), 8, 1),              # it did not: a crew takes it, CTAs the rest
    (((7, 1), (3, 8000)), 8, 1),
    (((7, 1), (3, 20000)), 8, 0),               # the launch takes as long anyway
    (((7, 0), (3, 20000)), 8, 0),
    (((11, 47), (7, 2376), (5, 3440)), 4, 47),  # three primes: the crews take the largest
    (((11, 1), (7, 9), (5, 13)), 8, 10),        # few quartics of any prime: those of p >= 7
    (((11, 300), (5, 100)), 8, 0),              # many: one CTA each is the better split
    (((13, 2), (11, 20)), 8, 22),
])
def test_crews_take_the_heavy_quartics_of_a_mixed_launch(runtime, groups, crew, joint):
    kw = {f"{k}{i + 1}": v for i, g in enumerate(groups) for k, v in zip("pn", g)}
    assert runtime(op="joint", crew=crew, ctas=304, **kw)["rc"] == joint


def test_mixed_launch_is_one_launch(runtime):
    r = runtime(op="heights", p1=5, n1=65536, p2=11, n2=1)
    assert [f["crew"] for f in r["fused"]] == [8] and r["fused"][0]["grid"] == 304


@pytest.mark.parametrize("p,cta_bytes", [(7, 2 * 245904 * 4), (11, 2 * 5052676 * 4)])
def test_small_budgets_use_crews_only_while_each_quartic_gets_one(runtime, p, cta_bytes):
    # a crew of c takes a quartic in more than 1/c of a CTA's time: a second round of crews on a small grid is slower than
    # a CTA for each quartic (7 on a budget of 7 CTAs)
    for ctas in (1, 2, 3, 4, 5, 7, 8, 13, 40, 152, 200):
        r = runtime(op="heights", p1=p, n1=2 * ctas, budget=ctas * cta_bytes)
        assert r["rc"] == 0 and r["crews"][0] == ctas
        assert r["peak"] <= ctas * cta_bytes + 8000 + CONTROL_BYTES
        for n, crew in enumerate(r["crew_for"][:2 * ctas + 1]):
            assert n == 0 or crew == 1 or n <= r["crews"][crew.bit_length() - 1]
            if 1 <= n <= ctas // 2:
                assert crew > 1   # there is room for a crew of 2 for each
    # the whole device: two CTAs per SM share it, and up to three rounds of crews are faster
    r = runtime(op="heights", p1=p, n1=1000)
    assert r["crews"] == [304, 152, 76, 38]
    assert [r["crew_for"][n] for n in (1, 38, 39, 228, 229, 456, 457)] == [8, 8, 4, 4, 2, 2, 1]


def test_mixed_launch_on_a_small_budget_uses_its_ctas(runtime):
    for ctas in (1, 3, 7, 13, 40, 100):
        r = runtime(op="heights", p1=5, n1=3000, p2=11, n2=30, budget=ctas * 2 * 5052676 * 4)
        assert r["rc"] == 0 and len(r["fused"]) == 1
        assert r["fused"][0]["grid"] >= ctas - ctas // 8


CTA_BYTES = {p: 8 * w for p, w in {7: 245904, 11: 5052676, 13: 13138404}.items()}   # two chain buffers


@pytest.mark.parametrize("p,n", [(7, 1), (7, 20), (11, 3), (13, 1)])
def test_no_memory_for_crews_runs_without_them(runtime, p, n):
    # memory for a CTA per quartic, but not for the CTAs of a crew: the call runs as it did without crews
    limit = n * CTA_BYTES[p] + 8 * n + CONTROL_BYTES
    r = runtime(op="heights", p1=p, n1=n, limit=limit)
    assert r["rc"] == 0 and [f["crew"] for f in r["fused"]] == [1] and r["fused"][0]["grid"] == n
    assert runtime(op="heights", p1=p, n1=n, limit=CTA_BYTES[p] // 2)["rc"] == 5
    assert len(runtime(op="heights", p1=p, n1=n)["fused"]) > 1
    assert runtime(op="prepare", p=p, n=n, limit=limit)["rc"] == 0
    r = runtime(op="theta_matrix", p=p, n=n, limit=limit)
    assert r["rc"] == 0 and r["launches"] == [f"theta_matrix n={n} crew=1"]
    assert runtime(op="theta_matrix", p=p, n=n)["launches"] == [f"theta_matrix n={n} crew=8"]
    r = runtime(op="heights", p1=p, n1=n, p2=3, n2=2, limit=(n + 2) * CTA_BYTES[p] + 8 * (n + 2) + CONTROL_BYTES)
    assert r["rc"] == 0 and [f["crew"] for f in r["fused"]] == [1]


def test_products_and_powers_without_memory_for_all_at_once(runtime):
    # (the harness's scratch sizes: (n + m) k bytes, 4 MB per prime side by side)
    n, m, k = 20001, 7000, 9000
    r = runtime(op="matmul", n=n, m=m, k=k)
    assert r["launches"] == [f"matmul n={n} m={m} k={k} a={MB} c={MB}"]
    r = runtime(op="matmul", n=n, m=m, k=k, limit=13000 * k)
    done = 0
    for x in r["launches"]:
        rows, a, c = (int(re.search(rf"\b{key}=(\d+)", x).group(1)) for key in "nac")
        assert (a, c) == (MB + done * k, MB + done * m) and (rows + m) * k <= 13000 * k
        done += rows
    assert r["rc"] == 0 and done == n
    assert runtime(op="matmul", n=n, m=m, k=k, limit=m * k)["rc"] == 5
    assert runtime(op="poly_power")["launches"] == ["poly_power at_once=5"]
    assert runtime(op="poly_power", limit=19 * MB)["launches"] == ["poly_power at_once=1"]
    assert runtime(op="poly_power", limit=3 * MB)["rc"] == 5


def test_a_workspace_that_suffices_is_kept(runtime):
    # a call that would like crews, beside a workspace for one quartic: without memory for both it keeps the old one
    one = runtime(op="prepare", p=11, n=1)["live"]
    r = runtime(op="theta_matrix", p=7, n=30, after=11, limit=one + 20 * MB)
    assert r["rc"] == 0 and r["launches"] == ["theta_matrix n=30 crew=1"] and r["live"] <= one + MB


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("power", [0, 1, 2])
@pytest.mark.parametrize("p", [3, 5, 7, 11, 13])
def test_two_ctas_per_sm_in_every_mode(runtime, p, power, form):
    # the shared memory of a launch: two CTAs share an SM at every prime, and a form pays only for its own product
    r = runtime(op="heights", p1=p, n1=100000, power=power, form=form, max_ctas=10 ** 6)
    assert [f["grid"] for f in r["fused"]] == [2 * 152]
    if form == 0 and power == 2:   # nothing is staged: the iterates and the mode's byte arrays
        ld, fpm2, d1f = ((d + 1) * (d + 2) * (d + 3) // 6 for d in (4 * (p - 1), 4 * (p - 2), 4 * p))
        assert r["fused"][0]["smem"] <= 6000 + 2 * ld + fpm2 + d1f + 300


@pytest.mark.parametrize("form,thresholds", [(0, 7), (1, 1)])
def test_sweep_autotune_times_what_has_an_effect(runtime, form, thresholds):
    # one warm-up and two timed launches for each shape; the dp4a product runs every tap pair whatever the threshold
    r = runtime(op="sweep_autotune", form=form, p=5, n=20000)
    assert r["rc"] == 0
    assert r["launches"].count("screen") == 3 * thresholds * 2 and len(r["fused"]) == 3 * thresholds * 2
    assert r["launches"][-1].startswith("best dense_min=0 ")
