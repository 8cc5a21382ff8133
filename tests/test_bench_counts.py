"""The transforms that bench.py's rooflines take a step to launch, against a walk through what the library enqueues."""
from types import SimpleNamespace

import pytest

import bench
from paper_2606_17421_b200 import workloads as wl

FUSED_STAGES = 8        # of a digit's transform, where its second pass is part of the key-switch product


def walk(r, n_in, n_out, b, g, double, per_output):
    """Forward and inverse transforms of one call: lists of (modulus index, part of the stages)."""
    fwd, inv = [], []

    def digits(own_prime, in_product, logn):
        for digit in range(r):
            for m in range(r + 1):
                if m == digit and not own_prime:
                    continue                            # its transform is at hand
                fwd.append((m, 1 - FUSED_STAGES / logn if in_product else 1))

    for q in range(n_in):
        fwd += [(m, 1) for m in range(r)] * 2
        if b > 1:
            digits(False, not double, 15)
        if not double:
            for k in range(1, b):
                for comp in range(2):
                    inv.append((r, 1))                  # the residue modulo P, whose lift is transformed into every prime
                    fwd += [(m, 1) for m in range(r)]
    for p in range(n_out):
        for j in range(1, g):
            inv += [(m, 1) for m in range(r + 1 if double else r)]
            digits(double, True, 15)
        for comp in range(2):
            inv += [(m, 1) for m in range(r)]
            if g > 1:
                inv += [(r, 1)] * (1 if per_output else g - 1)
            if double:
                inv += [(r, 1)] * (g if comp == 0 else 1)
    return fwd, inv


@pytest.mark.parametrize("b,g", [(16, 4), (64, 1), (1, 64), (8, 8)])
@pytest.mark.parametrize("hoist", ["single", "double"])
@pytest.mark.parametrize("moddown", ["per_rotation", "per_output"])
def test_transform_counts_follow_what_a_call_enqueues(b, g, hoist, moddown):
    ps = wl.PARAM_SETS["n15"]
    n_in, n_out = 2, 3
    run = SimpleNamespace(r=7, N=1 << 15, primes=ps["primes"], P=ps["special"], layers=[dict(n_in=n_in, n_out=n_out, b=b, g=g)],
                          plan=SimpleNamespace(hoist=hoist, moddown=moddown), transforms_weights_per_call=lambda e: False)
    got = bench.transform_counts(run)
    fwd, inv = walk(7, n_in, n_out, b, g, hoist == "double", moddown == "per_output")
    for name, launched in (("fwd", fwd), ("inv", inv)):
        assert got[name]["polys"] == pytest.approx(sum(part for _, part in launched), abs=0.06), name
        assert got[name]["fp64_polys"] == pytest.approx(sum(part for m, part in launched if m < 7), abs=0.06), name


def test_transform_counts_of_one_projection():
    # 768 -> 2304 without flags, modulo each ciphertext prime: the input 2, digits 6 + 9 x 6, lifts 15 x 2; 8 of 15 stages of the digits
    # are counted with the key-switch products
    ps = wl.PARAM_SETS["n15"]
    run = SimpleNamespace(r=7, N=1 << 15, primes=ps["primes"], P=ps["special"], layers=[dict(n_in=1, n_out=3, b=16, g=4)],
                          plan=SimpleNamespace(hoist="single", moddown="per_rotation"), transforms_weights_per_call=lambda e: False)
    assert bench.transform_counts(run)["fwd"]["fp64_polys"] == 7 * (92 - 60 * 8 / 15)
