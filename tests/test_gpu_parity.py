"""GPU parity: every kernel family and every entry point of the C ABI against the CPU oracle,
bit for bit on every residue, on the same seeded inputs."""
import numpy as np
import pytest

from oracle import ckks
from paper_2606_17421_b200 import workloads as wl
from tests.helpers import GpuSide, custom_params, oracle_params

pytestmark = pytest.mark.gpu

# the plan variant the benchmark's headline runs: two row blocks per plaintext, one division by P per output
# ciphertext, baby-step rotations kept in the extended basis
BEST = dict(pack="complex", moddown="per_output", hoist="double")


# ------------------------------------------------------------------ transforms

@pytest.mark.parametrize("logN,n_small", [(10, 1), (12, 2), (13, 3), (15, 6), (16, 8)])
def test_negacyclic_mul_matches_oracle(logN, n_small):
    N = 1 << logN
    par = custom_params(N, n_small)
    g = GpuSide(par, ckks.Plan(64, 1, 8, 8))
    try:
        nb = par.r + 1
        n_polys = 2 * nb + 3                      # not a whole number of basis groups
        rng = np.random.default_rng(logN)
        moduli = [par.basis[t % nb] for t in range(n_polys)]
        a = np.stack([rng.integers(0, q, size=N, dtype=np.uint64) for q in moduli])
        b = np.stack([rng.integers(0, q, size=N, dtype=np.uint64) for q in moduli])
        a[0, :] = np.uint64(moduli[0] - 1)        # extreme residues
        b[0, :] = np.uint64(moduli[0] - 1)
        a[1, :] = 0
        out = g.empty_u64(n_polys, N)
        g.bf.bf_negacyclic_mul(g.ctx, g.to_dev(a), g.to_dev(b), out, n_polys)
        expect = ckks.ring_mul(a, b, moduli, par)
        assert np.array_equal(g.to_host_u64(out), expect)
    finally:
        g.close()


# ------------------------------------------------------------------ encoder

ENCODE_CASES = [
    # param set / ring, plan, (d_out, d_in)
    ("n12", (64, 1, 8, 8), (64, 64)),
    ("n12", (64, 4, 4, 4), (100, 130)),          # ragged: zero padding in rows and columns
    ("n12", (256, 8, 8, 4), (300, 256)),
    ("n15", (1024, 16, 8, 8), (1100, 768)),
]


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("pack", ["real", "complex"])
@pytest.mark.parametrize("pkey,plan_t,shape", ENCODE_CASES)
def test_encode_weights_matches_oracle(pkey, plan_t, shape, compact, pack):
    par = oracle_params(pkey)
    plan = ckks.Plan(*plan_t, pack=pack)
    d_out, d_in = shape
    W = wl.gen_weights(1, f"enc{pkey}{plan_t}", d_out, d_in)
    g = GpuSide(par, plan)
    try:
        g.bf.bf_set_compact_cache(g.ctx, compact)
        w = g.bf.bf_encode_weights(g.ctx, g.to_dev(W), d_out, d_in)
        n_in, n_out = -(-d_in // plan.D), plan.n_out(d_out)
        used = g.bf.bf_cache_bytes_used(g.ctx)
        assert used == g.bf.bf_weights_bytes(g.ctx, d_out, d_in)
        # every encoded word is resident once: 8 bytes, or in the compact cache the narrowest format its
        # prime allows (4, 5 or 8 bytes); layout padding comes on top
        word_bytes = sum(4 if q < 2 ** 32 else 5 if q < 2 ** 40 else 8 for q in par.primes) if compact else 8 * par.r
        words = n_in * n_out * plan.M * par.N
        assert words * word_bytes <= used
        if compact and word_bytes < 8 * par.r:
            g.bf.bf_set_compact_cache(g.ctx, False)
            assert used < g.bf.bf_weights_bytes(g.ctx, d_out, d_in)
            g.bf.bf_set_compact_cache(g.ctx, True)
        idx = [(p, q, j, k) for p in range(n_out) for q in range(n_in) for j in range(plan.g) for k in range(plan.b)]
        if len(idx) > 48:                         # sample, always keeping the corners
            rng = np.random.default_rng(0)
            keep = {0, len(idx) - 1} | set(rng.choice(len(idx), 46, replace=False).tolist())
            idx = [idx[i] for i in sorted(keep)]
        out = g.empty_u64(par.r, par.N)
        for (p, q, j, k) in idx:
            z = ckks.plain_slots(W, plan, p, q, j, k, par.n)
            expect = ckks.to_residues(ckks.encode_coeffs(z, par.N, par.scale), par.primes)
            g.bf.bf_weights_export(g.ctx, w, p, q, j, k, out)
            assert np.array_equal(g.to_host_u64(out), expect), (p, q, j, k)
        g.bf.bf_weights_free(g.ctx, w)
        assert g.bf.bf_cache_bytes_used(g.ctx) == 0
    finally:
        g.close()


@pytest.mark.parametrize("d_out,plan_t", [(16, (16, 1, 16, 1)), (16, (16, 1, 8, 2)), (40, (16, 1, 16, 1)), (100, (16, 1, 4, 4))])
def test_weights_of_few_output_groups_count_for_their_words_only(d_out, plan_t):
    # 1, 2, 3 and 28 groups, where a small ring's tiles have 8 lanes: idle lanes are neither counted nor, where one stage has
    # them all, stored
    import torch
    par, plan = oracle_params("n12"), ckks.Plan(*plan_t)
    g = GpuSide(par, plan)
    try:
        W = torch.randn(d_out, 16 * 40, device="cuda") * 0.02
        groups, terms = plan.n_out(d_out) * plan.g, 40 * plan.b
        widths = {False: 8 * par.r, True: sum(5 if q < 2 ** 40 else 8 for q in par.primes)}
        for compact in (False, True):
            g.bf.bf_set_compact_cache(g.ctx, compact)
            assert g.bf.bf_weights_bytes(g.ctx, d_out, 16 * 40) == widths[compact] * par.N * groups * terms
        g.bf.bf_weights_free(g.ctx, g.bf.bf_encode_weights(g.ctx, W, d_out, 16 * 40))       # (scratch, code)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        handles = [g.bf.bf_encode_weights(g.ctx, W, d_out, 16 * 40) for _ in range(4)]
        stored = (free - torch.cuda.mem_get_info()[0]) / 4
        assert stored <= widths[True] * par.N * (groups if groups <= 8 else groups + 4) * terms + (3 << 20)
        assert len(handles) == 4
    finally:
        g.close()


# ------------------------------------------------------------------ key switch, rescale

@pytest.mark.parametrize("pkey", ["n12", "n15"])
def test_rotate_matches_oracle(pkey):
    par = oracle_params(pkey)
    plan = ckks.Plan(64, 1, 8, 8) if pkey == "n12" else ckks.Plan(1024, 16, 4, 16)
    s = ckks.keygen(par, 3)
    keys = ckks.make_rotation_keys(par, s, plan, 3)
    g = GpuSide(par, plan)
    try:
        steps = g.load_keys(keys)
        rng = np.random.default_rng(7)
        z = rng.normal(size=par.n)
        ct = ckks.encrypt(par, s, ckks.encode_coeffs(z, par.N, par.scale), 4)
        out = g.empty_u64(2, par.r, par.N)
        for st in steps[:4] + steps[-2:]:
            g.bf.bf_rotate(g.ctx, g.to_dev(ct), st, out)
            expect = ckks.rotate(par, ct, st, keys)
            got = g.to_host_u64(out)
            assert np.array_equal(got, expect), st
            dec = ckks.decode(ckks.decrypt(par, s, got), par.N, par.scale)
            assert np.abs(dec - np.roll(z, -st)).max() < 1e-6
        with pytest.raises(g.bf.BifrostError) as ei:
            g.bf.bf_rotate(g.ctx, g.to_dev(ct), 12345, out)
        assert ei.value.code == g.bf.BF_ERR_MISSING_KEY
    finally:
        g.close()


@pytest.mark.parametrize("logN,n_primes", [(10, 2), (10, 5), (11, 8), (10, 10), (10, 15)])
def test_rotate_for_every_arrangement_of_digits_in_a_block(logN, n_primes):
    # the fused transform and inner product of one rotation, a launch that does not fill the GPU: one chunk a block, idle warps, a warp
    # per digit, digits in two rounds of 8 warps (several chunks a block: see the folds of many ciphertexts)
    par = ckks.Params(1 << logN, ckks.find_primes(1 << 40, 2 << logN, n_primes), ckks.find_primes(1 << 60, 2 << logN, 1)[0], 2.0 ** 30)
    plan = ckks.Plan(8, 1, 4, 2)
    s = ckks.keygen(par, 5)
    keys = ckks.make_rotation_keys(par, s, plan, 5)
    g = GpuSide(par, plan)
    try:
        steps = g.load_keys(keys)
        ct = ckks.encrypt(par, s, ckks.encode_coeffs(np.arange(par.n) % 7 - 3.0, par.N, par.scale), 6)
        out = g.empty_u64(2, par.r, par.N)
        for st in (steps[0], steps[-1]):
            g.bf.bf_rotate(g.ctx, g.to_dev(ct), st, out)
            assert np.array_equal(g.to_host_u64(out), ckks.rotate(par, ct, st, keys)), st
    finally:
        g.close()


@pytest.mark.parametrize("n_primes", [3, 4, 6, 7, 9, 11, 12, 13, 14])
def test_rotate_for_the_other_digit_counts(n_primes):
    # (an instance of the fused transform and inner product each)
    test_rotate_for_every_arrangement_of_digits_in_a_block(10, n_primes)


@pytest.mark.parametrize("pkey", ["n12", "n15"])
def test_rescale_matches_oracle(pkey):
    par = oracle_params(pkey)
    g = GpuSide(par, ckks.Plan(64, 1, 8, 8))
    try:
        rng = np.random.default_rng(8)
        cts = np.stack([np.stack([ckks.sample_uniform(rng, par.primes, par.N) for _ in range(2)]) for _ in range(3)])
        cts[0, 0, -1, :5] = [0, 1, (par.primes[-1] - 1) // 2, (par.primes[-1] - 1) // 2 + 1, par.primes[-1] - 1]
        expect = np.stack([ckks.rescale(par, c) for c in cts])
        d_in = g.to_dev(cts)
        d_out = g.empty_u64(3, 2, par.r - 1, par.N)
        new_scale = g.bf.bf_rescale(g.ctx, d_in, d_out, 3, par.r, par.scale * par.scale)
        assert np.array_equal(g.to_host_u64(d_out), expect)
        assert new_scale == par.scale * par.scale / par.primes[-1]
        # in place, several ciphertexts
        g.bf.bf_rescale(g.ctx, d_in, d_in, 3, par.r)
        flat = g.to_host_u64(d_in).reshape(-1)[:expect.size].reshape(expect.shape)
        assert np.array_equal(flat, expect)
        # a second level down, from the packed output
        expect2 = np.stack([ckks.rescale(par, c) for c in expect])
        d2 = g.empty_u64(3, 2, par.r - 2, par.N)
        if par.r - 1 >= 2:
            g.bf.bf_rescale(g.ctx, d_out, d2, 3, par.r - 1)
            assert np.array_equal(g.to_host_u64(d2), expect2)
        with pytest.raises(g.bf.BifrostError) as ei:
            g.bf.bf_rescale(g.ctx, d_in, d_in, 1, 1)
        assert ei.value.code == g.bf.BF_ERR_LEVEL
    finally:
        g.close()


# ------------------------------------------------------------------ the linear layer

def run_case(par, plan, d_out, d_in, seed, tol, tag, tight=1e-5):
    W = wl.gen_weights(seed, tag, d_out, d_in)
    x = wl.gen_activation(seed, tag, d_in)
    s = ckks.keygen(par, seed)
    keys = ckks.make_rotation_keys(par, s, plan, seed)
    cts = ckks.encrypt_vector(par, plan, s, x, seed)
    expect = ckks.linear(par, plan, cts, W, keys)
    n_out = plan.n_out(d_out)
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        Wd = g.to_dev(W)
        w = g.bf.bf_encode_weights(g.ctx, Wd, d_out, d_in)
        got_cached = g.to_host_u64(g.linear(cts, W, d_out, d_in, weights=w))
        got_fallback = g.to_host_u64(g.linear(cts, W, d_out, d_in, weights=None))
        for p in range(n_out):
            assert np.array_equal(got_cached[p], expect[p]), ("cached", p)
            assert np.array_equal(got_fallback[p], expect[p]), ("fallback", p)
        # the configuration the benchmark times: the same buffers again and again, so that the call is
        # captured and then replayed as a graph with its concurrent key-switch lanes
        ct_in = g.to_dev(np.stack(cts))
        ct_out = g.empty_u64(n_out, 2, par.r, par.N)
        for call in range(4):
            ct_out.zero_()
            g.bf.bf_linear(g.ctx, ct_in, len(cts), w, None, d_out, d_in, ct_out, n_out)
        got_replayed = g.to_host_u64(ct_out)
        for p in range(n_out):
            assert np.array_equal(got_replayed[p], expect[p]), ("replayed", p)
        # the compact cache format (narrower words per prime) changes no residue, cached or on the fly
        g.bf.bf_set_compact_cache(g.ctx, True)
        w_compact = g.bf.bf_encode_weights(g.ctx, Wd, d_out, d_in)
        got_compact = g.to_host_u64(g.linear(cts, W, d_out, d_in, weights=w_compact))
        got_compact_fallback = g.to_host_u64(g.linear(cts, W, d_out, d_in, weights=None))
        got_mixed = g.to_host_u64(g.linear(cts, W, d_out, d_in, weights=w))        # the older handle still works
        g.bf.bf_set_compact_cache(g.ctx, False)
        for p in range(n_out):
            assert np.array_equal(got_compact[p], expect[p]), ("compact", p)
            assert np.array_equal(got_compact_fallback[p], expect[p]), ("compact fallback", p)
            assert np.array_equal(got_mixed[p], expect[p]), ("mixed", p)
        g.bf.bf_weights_free(g.ctx, w_compact)
        # rescale on the device, decrypt on the host, compare with the fp64 product
        d_ct = g.to_dev(got_cached)
        low = g.empty_u64(n_out, 2, par.r - 1, par.N)
        scale = g.bf.bf_rescale(g.ctx, d_ct, low, n_out, par.r, par.scale * par.scale)
        low = g.to_host_u64(low)
        y = np.zeros(d_out)
        for p in range(n_out):
            assert np.array_equal(low[p], ckks.rescale(par, expect[p]))
            part = ckks.fold_output(ckks.decode(ckks.decrypt(par, s, low[p]), par.N, scale), plan, p, d_out)
            y[p * plan.rows_per_ct:p * plan.rows_per_ct + len(part)] = part
        err = np.abs(y - W.astype(np.float64) @ x).max()
        assert err < tol, err
        assert err < tight         # far inside the stated tolerance; catches scale bookkeeping slips
        # the host-buffer entry point gives the same rescaled ciphertexts
        import torch
        h_in = torch.from_numpy(np.stack(cts).view(np.int64)).pin_memory()
        h_out = torch.empty((n_out, 2, par.r - 1, par.N), dtype=torch.int64).pin_memory()
        g.bf.bf_linear_host(g.ctx, h_in, len(cts), w, None, d_out, d_in, h_out, n_out)
        assert np.array_equal(h_out.numpy().view(np.uint64), low)
        # product and rescale as one call: cached (direct, captured, replayed) and on the fly
        low_fused = g.empty_u64(n_out, 2, par.r - 1, par.N)
        for call in range(3):
            low_fused.zero_()
            assert g.bf.bf_linear_rescaled(g.ctx, ct_in, len(cts), w, None, d_out, d_in, low_fused, n_out,
                                           par.scale * par.scale) == scale
        assert np.array_equal(g.to_host_u64(low_fused), low)
        low_fused.zero_()
        g.bf.bf_linear_rescaled(g.ctx, ct_in, len(cts), None, Wd, d_out, d_in, low_fused, n_out)
        assert np.array_equal(g.to_host_u64(low_fused), low)
        # the two entry points on the SAME output address (replayed launch sequences are keyed by the arguments):
        # a full-level result, then a rescaled one, then a full-level one again, each repeated into its replay
        shared = g.empty_u64(n_out, 2, par.r, par.N)
        shared_low = shared.view(-1)[:n_out * 2 * (par.r - 1) * par.N].view(n_out, 2, par.r - 1, par.N)
        for kind in ("full", "rescaled", "full"):
            for call in range(3):
                shared.zero_()
                if kind == "full":
                    g.bf.bf_linear(g.ctx, ct_in, len(cts), w, None, d_out, d_in, shared, n_out)
                else:
                    g.bf.bf_linear_rescaled(g.ctx, ct_in, len(cts), w, None, d_out, d_in, shared_low, n_out)
            if kind == "full":
                assert np.array_equal(g.to_host_u64(shared), got_cached), kind
            else:
                assert np.array_equal(g.to_host_u64(shared_low), low), kind
    finally:
        g.close()


def test_linear_tiny_config_bit_exact():
    w = wl.WORKLOADS["tiny"]
    par = oracle_params(w.params)
    run_case(par, ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g), 64, 64, 0, 1e-2, "tiny")


@pytest.mark.parametrize("plan_t,shape", [
    ((64, 4, 4, 4), (100, 130)),      # tau > 1, ragged rows and columns, 2 x 3 tiles
    ((64, 32, 2, 1), (64, 64)),       # fully dense packing, no giant step
    ((128, 1, 1, 128), (128, 128)),   # no baby step: every diagonal its own giant rotation
    ((32, 1, 32, 1), (40, 32)),       # all rotations hoisted from the input
    ((32, 32, 1, 1), (70, 50)),       # one diagonal per tile: no rotation at all, 3 x 2 tiles
    ((64, 4, 16, 1), (150, 64)),      # 16 terms per output group, odd number of groups: half-filled last stage
    ((64, 4, 4, 4), (64, 1472)),      # 23 input chunks: their 69 baby rotations span two key-switch batches
    ((64, 4, 4, 4), (1920, 64)),      # 30 output blocks: their 90 giant rotations span two key-switch batches
])
def test_linear_small_ring_plans(plan_t, shape):
    par = oracle_params("n12")
    run_case(par, ckks.Plan(*plan_t), shape[0], shape[1], 2, 1e-2, f"small{plan_t}")


@pytest.mark.parametrize("plan_t,shape", [
    ((64, 4, 4, 4), (100, 130)),      # two row blocks -> one output ciphertext, ragged second block
    ((64, 4, 4, 4), (150, 64)),       # three row blocks -> two ciphertexts, the last one with an empty imaginary part
    ((64, 1, 8, 8), (128, 64)),       # classical replicated layout, both parts full
    ((32, 32, 1, 1), (70, 50)),       # no rotation at all
    ((64, 4, 4, 4), (1920, 64)),      # 15 output ciphertexts
])
def test_linear_complex_packing_small_ring(plan_t, shape):
    par = oracle_params("n12")
    run_case(par, ckks.Plan(*plan_t, pack="complex"), shape[0], shape[1], 6, 1e-2, f"cplx{plan_t}")


def test_linear_gpt2_qkv_complex_packing_bit_exact():
    # the 768 -> 2304 projection with two row blocks per plaintext: 2 output ciphertexts instead of 3
    w = wl.WORKLOADS["gpt2_qkv"]
    par = oracle_params(w.params)
    L = w.layers[0]
    run_case(par, ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g, pack="complex"), L.d_out, L.d_in, 0, 1e-3, L.name)


@pytest.mark.parametrize("pack", ["real", "complex"])
@pytest.mark.parametrize("plan_t,shape", [
    ((64, 4, 4, 4), (100, 130)),      # three giant rotations per output, two or one output ciphertexts
    ((64, 1, 8, 8), (128, 64)),       # seven giant rotations per output
    ((64, 1, 2, 32), (64, 64)),       # 31 giant rotations summed before the one division
    ((64, 32, 2, 1), (64, 64)),       # no giant step: nothing to merge
    ((64, 4, 4, 4), (1920, 64)),      # 90 (45) giant rotations: several key-switch launches feed one division stage
])
def test_linear_one_division_by_P_per_output_small_ring(plan_t, shape, pack):
    par = oracle_params("n12")
    run_case(par, ckks.Plan(*plan_t, pack=pack, moddown="per_output"), shape[0], shape[1], 7, 1e-2, f"po{plan_t}")


@pytest.mark.parametrize("pack", ["real", "complex"])
def test_linear_gpt2_qkv_one_division_by_P_per_output_bit_exact(pack):
    w = wl.WORKLOADS["gpt2_qkv"]
    par = oracle_params(w.params)
    L = w.layers[0]
    plan = ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g, pack=pack, moddown="per_output")
    run_case(par, plan, L.d_out, L.d_in, 0, 1e-3, L.name)


@pytest.mark.parametrize("pack,moddown", [("real", "per_rotation"), ("complex", "per_output")])
@pytest.mark.parametrize("plan_t,shape", [
    ((64, 4, 4, 4), (100, 130)),      # three input ciphertexts, ragged
    ((64, 1, 8, 8), (128, 64)),       # classical layout, seven baby rotations
    ((64, 32, 2, 1), (64, 64)),       # no giant step
    ((128, 1, 1, 128), (128, 128)),   # no baby step: only P * ct, whose division by P is exact
    ((64, 4, 16, 1), (150, 64)),      # 16 terms per group, half-filled last stage
    ((64, 4, 4, 4), (64, 1472)),      # 23 input ciphertexts: their baby rotations span two key-switch batches
])
def test_linear_double_hoisting_small_ring(plan_t, shape, pack, moddown):
    if plan_t[3] - 1 > 64 and moddown == "per_output":
        pytest.skip("per-output division sums at most 64 giant steps")
    par = oracle_params("n12")
    run_case(par, ckks.Plan(*plan_t, pack=pack, moddown=moddown, hoist="double"), shape[0], shape[1], 8, 1e-2, f"dh{plan_t}")


@pytest.mark.parametrize("pack,moddown", [("real", "per_rotation"), ("complex", "per_output")])
def test_linear_gpt2_qkv_double_hoisting_bit_exact(pack, moddown):
    w = wl.WORKLOADS["gpt2_qkv"]
    par = oracle_params(w.params)
    L = w.layers[0]
    plan = ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g, pack=pack, moddown=moddown, hoist="double")
    run_case(par, plan, L.d_out, L.d_in, 0, 1e-3, L.name)


def test_linear_double_hoisting_with_the_papers_own_parameter_set():
    # a 60-bit ciphertext prime next to the 60-bit special prime: whole-word accumulation for every prime
    par = oracle_params("paper_n13")
    run_case(par, ckks.Plan(256, 16, 4, 4, hoist="double"), 300, 520, 4, 1e-2, "paper_n13_dh", tight=1e-3)


@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("modes", [{}, BEST], ids=["plain", "best"])
def test_weights_kept_as_coefficients_give_the_same_ciphertexts(bits, modes):
    # the coefficient form of the cache: rounded integer coefficients are resident, reduced per prime and
    # transformed on every call; residues must not change, and the handle is 1/r (1/2r) of the usual size
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4, **modes)
    d_out, d_in = 150, 130
    s = ckks.keygen(par, 61)
    keys = ckks.make_rotation_keys(par, s, plan, 61)
    W = wl.gen_weights(61, "coef", d_out, d_in)
    if bits == 32:      # on this small ring the slot vectors repeat eight times, which concentrates the coefficients:
        W = W / 32      # keep them inside 32 bits (the full-size rings have no replication and fit as they are)
    cts = ckks.encrypt_vector(par, plan, s, wl.gen_activation(61, "coef", d_in), 61)
    expect = ckks.linear(par, plan, cts, W, keys)
    n_out, n_in = plan.n_out(d_out), 3
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        Wd = g.to_dev(W)
        full_bytes = g.bf.bf_weights_bytes(g.ctx, d_out, d_in)
        g.bf.bf_set_coefficient_cache(g.ctx, bits)
        w = g.bf.bf_encode_weights(g.ctx, Wd, d_out, d_in)
        used = g.bf.bf_cache_bytes_used(g.ctx)
        assert used == n_in * n_out * plan.M * par.N * bits // 8 == g.bf.bf_weights_bytes(g.ctx, d_out, d_in)
        assert used * par.r * (64 // bits) <= full_bytes
        ct_in = g.to_dev(np.stack(cts))
        ct_out = g.empty_u64(n_out, 2, par.r, par.N)
        for call in range(4):                       # direct, captured, replayed
            ct_out.zero_()
            g.bf.bf_linear(g.ctx, ct_in, n_in, w, None, d_out, d_in, ct_out, n_out)
            got = g.to_host_u64(ct_out)
            for p in range(n_out):
                assert np.array_equal(got[p], expect[p]), (call, p)
        out = g.empty_u64(par.r, par.N)
        for (p, q, j, k) in ((0, 0, 0, 0), (n_out - 1, 2, 3, 1), (0, 1, 2, 3)):
            z = ckks.plain_slots(W, plan, p, q, j, k, par.n)
            g.bf.bf_weights_export(g.ctx, w, p, q, j, k, out)
            assert np.array_equal(g.to_host_u64(out), ckks.to_residues(ckks.encode_coeffs(z, par.N, par.scale), par.primes))
        # a transform-domain handle made afterwards works beside it
        g.bf.bf_set_coefficient_cache(g.ctx, 0)
        w2 = g.bf.bf_encode_weights(g.ctx, Wd, d_out, d_in)
        got = g.to_host_u64(g.linear(cts, W, d_out, d_in, weights=w2))
        assert all(np.array_equal(got[p], expect[p]) for p in range(n_out))
        g.bf.bf_weights_free(g.ctx, w)
        g.bf.bf_weights_free(g.ctx, w2)
        assert g.bf.bf_cache_bytes_used(g.ctx) == 0
        if bits == 32:      # coefficients beyond 32 bits are refused at encoding time
            g.bf.bf_set_coefficient_cache(g.ctx, 32)
            with pytest.raises(g.bf.BifrostError) as ei:
                g.bf.bf_encode_weights(g.ctx, g.to_dev(W * 1024), d_out, d_in)
            assert ei.value.code == g.bf.BF_ERR_RANGE
            assert g.bf.bf_cache_bytes_used(g.ctx) == 0
        with pytest.raises(g.bf.BifrostError):
            g.bf.bf_set_coefficient_cache(g.ctx, 16)
    finally:
        g.close()


def test_per_output_division_refuses_more_giant_steps_than_its_interface_allows():
    from paper_2606_17421_b200 import bifrost as bf
    ps = wl.PARAM_SETS["n12"]
    basis = list(ps["primes"]) + [ps["special"]]
    with pytest.raises(bf.BifrostError) as ei:          # g - 1 = 127 > 64
        bf.bf_ctx_create(ps["N"], basis, 3, 2.0 ** 40, bf.bf_plan(128, 1, 1, 128, bf.BF_PLAN_MODDOWN_PER_OUTPUT))
    assert ei.value.code == bf.BF_ERR_SHAPE
    with pytest.raises(bf.BifrostError) as ei:          # unknown flag bit
        bf.bf_ctx_create(ps["N"], basis, 3, 2.0 ** 40, bf.bf_plan(64, 1, 8, 8, 64))
    assert ei.value.code == bf.BF_ERR_INVALID_ARG


@pytest.mark.parametrize("modes", [{}, BEST, dict(hoist="double")], ids=["plain", "best", "double_hoist"])
def test_weights_with_a_split_of_their_own(modes):
    # one context (plan 8 x 4), three handles for the same matrix with the splits 8 x 4, 16 x 2 and 2 x 16, and a
    # coefficient-form handle with 4 x 8: every call matches the oracle run under that split; what the context
    # refuses: a split whose product is not D / tau, one that is not a power of two, a missing key
    from paper_2606_17421_b200 import bifrost as bf
    par = oracle_params("n12")
    base = ckks.Plan(64, 2, 8, 4, **modes)
    d_out, d_in, seed = 150, 100, 21
    W = wl.gen_weights(seed, "split", d_out, d_in)
    x = wl.gen_activation(seed, "split", d_in)
    s = ckks.keygen(par, seed)
    variants = [(8, 4), (16, 2), (2, 16), (4, 8)]
    plans = [ckks.Plan(base.D, base.tau, b, g, base.pack, base.moddown, base.hoist) for b, g in variants]
    extra = sorted({st for pl in plans for st in ckks.required_rotations(pl)})
    keys = ckks.make_rotation_keys(par, s, base, seed, extra_steps=extra)
    cts = ckks.encrypt_vector(par, base, s, x, seed)
    g = GpuSide(par, base)
    try:
        Wd = g.to_dev(W)
        g.load_keys(keys)                            # the keys of the plan's own split only
        w = g.bf.bf_encode_weights_split(g.ctx, Wd, d_out, d_in, 16, 2)
        with pytest.raises(bf.BifrostError) as ei:
            g.linear(cts, W, d_out, d_in, weights=w)
        assert ei.value.code == bf.BF_ERR_MISSING_KEY
        g.bf.bf_weights_free(g.ctx, w)
        g.load_keys(keys, extra_steps=extra)
        for bad in ((8, 8), (3, 11), (0, 32), (32, 0)):
            with pytest.raises(bf.BifrostError) as ei:
                g.bf.bf_encode_weights_split(g.ctx, Wd, d_out, d_in, *bad)
            assert ei.value.code == bf.BF_ERR_SHAPE, bad
        for (b, gg), plan in zip(variants, plans):
            expect = ckks.linear(par, plan, cts, W, keys)
            if (b, gg) == (4, 8):
                g.bf.bf_set_coefficient_cache(g.ctx, 64)
            w = g.bf.bf_encode_weights_split(g.ctx, Wd, d_out, d_in, b, gg)
            g.bf.bf_set_coefficient_cache(g.ctx, 0)
            n_out = plan.n_out(d_out)
            ct_in = g.to_dev(np.stack(cts))
            out = g.empty_u64(n_out, 2, par.r, par.N)
            for call in range(3):               # direct, captured, replayed
                out.zero_()
                g.bf.bf_linear(g.ctx, ct_in, len(cts), w, None, d_out, d_in, out, n_out)
            got = g.to_host_u64(out)
            for p in range(n_out):
                assert np.array_equal(got[p], expect[p]), (b, gg, p)
            g.bf.bf_weights_free(g.ctx, w)
    finally:
        g.close()


@pytest.mark.parametrize("case", range(32))
def test_random_small_ring_cases(case):
    # seeded random draws over what the other cases fix by hand: tile side, replica split, baby/giant split of the plan
    # and of the handle, the three plan flags, ragged shapes with one to three input and output blocks; the cached
    # call, the replayed call and the fused product + rescale must all match the oracle
    rng = np.random.default_rng(1000 + case)
    par = oracle_params("n12")
    D = int(rng.choice([32, 64, 128]))
    tau = int(rng.choice([t for t in (1, 2, 4, 8, 16) if D * t <= par.n and D // t >= 2]))
    M = D // tau
    splits = [(b, M // b) for b in (1, 2, 4, 8, 16, 32, 64) if b <= M and M % b == 0 and b - 1 <= 64 and M // b - 1 <= 64]
    b, g_ = splits[int(rng.integers(len(splits)))]
    hb, hg = splits[int(rng.integers(len(splits)))]
    modes = dict(pack=str(rng.choice(["real", "complex"])), moddown=str(rng.choice(["per_rotation", "per_output"])),
                 hoist=str(rng.choice(["single", "double"])))
    d_in = int(rng.integers(1, 3 * D + 1))
    d_out = int(rng.integers(1, 3 * D + 1))
    base = ckks.Plan(D, tau, b, g_, **modes)
    hplan = ckks.Plan(D, tau, hb, hg, **modes)
    seed = 2000 + case
    W = wl.gen_weights(seed, "rand", d_out, d_in)
    x = wl.gen_activation(seed, "rand", d_in)
    s = ckks.keygen(par, seed)
    extra = ckks.required_rotations(hplan)
    keys = ckks.make_rotation_keys(par, s, base, seed, extra_steps=extra)
    cts = ckks.encrypt_vector(par, base, s, x, seed)
    expect_base = ckks.linear(par, base, cts, W, keys)
    expect_h = ckks.linear(par, hplan, cts, W, keys)
    n_out = base.n_out(d_out)
    g = GpuSide(par, base)
    try:
        g.load_keys(keys, extra_steps=extra)
        Wd = g.to_dev(W)
        ct_in = g.to_dev(np.stack(cts))
        for plan, expect, w in ((base, expect_base, g.bf.bf_encode_weights(g.ctx, Wd, d_out, d_in)),
                                (hplan, expect_h, g.bf.bf_encode_weights_split(g.ctx, Wd, d_out, d_in, hb, hg))):
            out = g.empty_u64(n_out, 2, par.r, par.N)
            low = g.empty_u64(n_out, 2, par.r - 1, par.N)
            for call in range(3):
                out.zero_()
                low.zero_()
                g.bf.bf_linear(g.ctx, ct_in, len(cts), w, None, d_out, d_in, out, n_out)
                g.bf.bf_linear_rescaled(g.ctx, ct_in, len(cts), w, None, d_out, d_in, low, n_out)
            got, got_low = g.to_host_u64(out), g.to_host_u64(low)
            for p in range(n_out):
                assert np.array_equal(got[p], expect[p]), (case, plan, p)
                assert np.array_equal(got_low[p], ckks.rescale(par, expect[p])), (case, plan, p, "rescaled")
            g.bf.bf_weights_free(g.ctx, w)
        fly = g.to_host_u64(g.linear(cts, W, d_out, d_in))          # on the fly: the plan's own split
        for p in range(n_out):
            assert np.array_equal(fly[p], expect_base[p]), (case, p, "on the fly")
    finally:
        g.close()


@pytest.mark.parametrize("n_out", [124, 126])
def test_one_division_per_output_with_many_outputs(n_out):
    par = oracle_params("n12")
    run_case(par, ckks.Plan(16, 1, 8, 2, moddown="per_output"), n_out * 16, 16, 37, 1e-2, "short", tight=1e-2)


@pytest.mark.parametrize("pkey,plan_t,n_in,modes", [
    ("n12", (16, 1, 1, 16), 125, {}),                       # the inputs' transforms: n_in x 2 components x 3 primes x 16 chunks
    ("n12", (16, 1, 1, 16), 126, {}),
    ("paper_n13", (32, 2, 16, 1), 3, {}),                   # baby rotations divided by P: 15 n_in x 2 x 4 primes x 32 chunks
    ("paper_n13", (32, 2, 16, 1), 4, {}),
    ("n12", (16, 1, 2, 8), 50, dict(hoist="double")),       # inputs and digits at once: n_in x 3 digits x 5 x 16 chunks
    ("n12", (16, 1, 2, 8), 51, dict(hoist="double")),
])
def test_forward_passes_on_both_sides_of_the_short_launches(pkey, plan_t, n_in, modes):
    # forward passes of up to 12000 chunks have 4 points a thread, longer ones 8
    run_case(oracle_params(pkey), ckks.Plan(*plan_t, **modes), plan_t[0], plan_t[0] * n_in, 37, 1e-2, "short", tight=1e-2)


@pytest.mark.parametrize("modes", [{}, dict(moddown="per_output", hoist="double")], ids=["plain", "extended"])
@pytest.mark.parametrize("logN,bits,plan_t,shape", [
    (10, [50, 45, 40, 30], (32, 2, 4, 4), (70, 90)),        # every operand class; 12 terms (a stage half empty), 3 inputs
    (10, [59, 45, 38, 20], (64, 1, 16, 4), (64, 40)),       # a base prime beyond 2^50: 45 bits in 30-bit limbs
    (11, [50] + [40] * 6, (32, 4, 2, 4), (33, 100)),        # 7 digits in registers; one key, four inputs in parts
    (11, [50] + [40] * 8, (32, 2, 8, 2), (20, 60)),         # 9 digits, one output block, 16 terms
    (12, [40, 40], (64, 8, 1, 8), (100, 64)),               # 2 digits, no baby step
])
def test_operand_classes_and_tile_edges(logN, bits, plan_t, shape, modes):
    taken, primes = {}, []
    for bt in bits:                                         # the largest primes below each power of two, all distinct
        found = ckks.find_primes(1 << bt, 2 << logN, bits.count(bt))
        primes.append(found[taken.setdefault(bt, 0)])
        taken[bt] += 1
    P = ckks.find_primes(1 << 60, 2 << logN, 1)[0]
    par = ckks.Params(1 << logN, primes, P, 2.0 ** 40)
    # (residues are compared exactly; the bound on the decrypted result only catches slips of scale or packing)
    run_case(par, ckks.Plan(*plan_t, **modes), shape[0], shape[1], 31, 1e-2, "classes", tight=1e-2)


@pytest.mark.parametrize("base", [50, 60], ids=["narrow", "wide"])
@pytest.mark.parametrize("n_primes", [2, 3, 4, 5, 6, 8, 10, 11, 12, 15])
def test_baby_steps_inside_the_product_for_every_digit_count(n_primes, base):
    # an instance for each count up to 11, a loop beyond, where all ciphertext primes are below 2^50 and where one is not (7 and 9
    # digits: see above)
    two_n = 2 << 10
    P, wide = ckks.find_primes(1 << 60, two_n, 2)
    primes = [wide if base == 60 else ckks.find_primes(1 << 50, two_n, 1)[0]] + ckks.find_primes(1 << 40, two_n, n_primes - 1)
    run_case(ckks.Params(1 << 10, primes, P, 2.0 ** 40), ckks.Plan(16, 1, 4, 4, **BEST), 40, 40, 41, 1e-2, "digits", tight=1e-2)


@pytest.mark.parametrize("moddown", ["per_rotation", "per_output"])
@pytest.mark.parametrize("plan_t", [(32, 2, 4, 4), (32, 4, 1, 8)], ids=["baby_steps", "none"])
@pytest.mark.parametrize("bits,special_bits", [
    ([50, 40, 40], 49),                     # the special prime below 2^50 among such primes: 25-bit limbs
    ([45, 40, 39], 41),                     # ... below 2^41, the transforms' lazily reduced path
    ([59, 45, 40], 45),                     # a ciphertext prime beyond 2^50: 30-bit limbs throughout
    ([50, 40, 40], 38),                     # fp64 operands, 5-byte words
    ([50, 40, 40], 31),                     # ... 4-byte words
])
def test_double_hoisting_with_a_special_prime_of_every_operand_class(bits, special_bits, plan_t, moddown):
    two_n = 2 << 10
    primes = [ckks.find_primes(1 << b, two_n, 2)[i] for i, b in enumerate(bits) if i < 2] + ckks.find_primes(1 << bits[2], two_n, 3)[2:]
    P = ckks.find_primes(1 << special_bits, two_n, 1)[0]
    assert len(set(primes + [P])) == 4
    # (a special prime below the digits' primes: the key switch adds noise of about q / P times the usual, far below 2^80)
    run_case(ckks.Params(1 << 10, primes, P, 2.0 ** 40), ckks.Plan(*plan_t, moddown=moddown, hoist="double"), 70, 90, 13, 1e-2,
             "special", tight=1e-2)


@pytest.mark.parametrize("n_primes,n_in", [(3, 70), (15, 240)])
def test_wide_inputs_take_no_more_scratch_than_the_batched_rotations(n_primes, n_in):
    # 70 inputs: their digits in two batches, then rotated inside the multiply-accumulate.  240 inputs, 15 digits: the digits of
    # all of them (15 x 16 polynomials each) and their intermediates would be 0.6 GB and more, far beyond the rotated inputs that
    # this saves: in batches of 64 digits and rotated inputs are 0.25 GB, and the rest of a call's scratch is below 0.1 GB
    import torch
    par = ckks.Params(1 << 10, ckks.find_primes(1 << 40, 2 << 10, n_primes), ckks.find_primes(1 << 60, 2 << 10, 1)[0], 2.0 ** 30)
    plan = ckks.Plan(4, 1, 2, 2, hoist="double", moddown="per_output")
    d_in, d_out = n_in * 4, 4
    s = ckks.keygen(par, 5)
    keys = ckks.make_rotation_keys(par, s, plan, 5)
    W, x = wl.gen_weights(5, "wide", d_out, d_in), wl.gen_activation(5, "wide", d_in)
    cts = ckks.encrypt_vector(par, plan, s, x, 5)
    expect = ckks.linear(par, plan, cts, W, keys)
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        w = g.bf.bf_encode_weights(g.ctx, g.to_dev(W), d_out, d_in)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        got = g.to_host_u64(g.linear(cts, W, d_out, d_in, weights=w))
        assert free - torch.cuda.mem_get_info()[0] < 500 << 20
        assert np.array_equal(got[0], expect[0])
    finally:
        g.close()


@pytest.mark.parametrize("plan_t,shape,modes", [
    ((128, 1, 2, 64), (130, 128), {}),              # 63 giant steps, two outputs: launches of several batches, 2 * 63 separate terms
    ((128, 1, 2, 64), (130, 128), dict(hoist="double")),
    ((128, 1, 2, 64), (130, 128), dict(moddown="per_output")),
    ((128, 1, 1, 128), (128, 100), {}),             # more giant steps than a launch has rotations (with one division per output
    ((128, 1, 1, 128), (128, 100), dict(hoist="double")),       # the library refuses them: see the test of its refusals)
    ((64, 8, 8, 1), (64, 64), {}),                  # none: nothing to assemble, or the inner sums alone
    ((64, 8, 8, 1), (64, 64), dict(hoist="double")),
    ((64, 8, 8, 1), (64, 64), dict(moddown="per_output")),
])
def test_output_assembly_for_few_and_many_giant_steps(plan_t, shape, modes):
    par = ckks.Params(1 << 10, ckks.find_primes(1 << 40, 2 << 10, 3), ckks.find_primes(1 << 60, 2 << 10, 1)[0], 2.0 ** 40)
    run_case(par, ckks.Plan(*plan_t, **modes), shape[0], shape[1], 19, 1e-2, "giants", tight=1e-2)


@pytest.mark.parametrize("bits,modes", [(40, {}), (55, dict(moddown="per_output")), (40, dict(hoist="double"))],
                         ids=["fp64", "integer_per_output", "fp64_double_hoist"])
def test_more_outputs_than_the_second_dimension_of_a_grid_holds(bits, modes):
    # 32770 output ciphertexts of two components: the division that ends them has 65540 polynomials
    par = ckks.Params(1 << 10, ckks.find_primes(1 << bits, 2 << 10, 2), ckks.find_primes(1 << 60, 2 << 10, 1)[0], 2.0 ** 30)
    plan = ckks.Plan(2, 1, 1, 2, **modes)
    d_out, d_in, n_out = 65539, 2, 32770
    s = ckks.keygen(par, 23)
    keys = ckks.make_rotation_keys(par, s, plan, 23)
    W = wl.gen_weights(23, "tall", d_out, d_in)
    cts = ckks.encrypt_vector(par, plan, s, wl.gen_activation(23, "tall", d_in), 23)
    sample = [0, 1, 32766, 32767, 32768, n_out - 1]
    expect = ckks.linear(par, plan, cts, W, keys, blocks=sample)
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        w = g.bf.bf_encode_weights(g.ctx, g.to_dev(W), d_out, d_in)
        out = g.linear(cts, W, d_out, d_in, weights=w)
        assert out.shape[0] == n_out
        low = g.empty_u64(n_out, 2, par.r - 1, par.N)
        g.bf.bf_linear_rescaled(g.ctx, g.to_dev(np.stack(cts)), 1, w, None, d_out, d_in, low, n_out)
        for p in sample:
            assert np.array_equal(g.to_host_u64(out[p]), expect[p]), p
            assert np.array_equal(g.to_host_u64(low[p]), ckks.rescale(par, expect[p])), ("rescaled", p)
    finally:
        g.close()


@pytest.mark.parametrize("bits", [(50, 40, 40), (60, 40, 30), (50,) + (40,) * 6], ids=["narrow", "wide", "seven_digits"])
@pytest.mark.parametrize("modes", [{}, BEST, dict(hoist="double")], ids=["plain", "best", "double_hoist"])
def test_tiles_of_16_coefficients(bits, modes):
    # 100 terms a group (the last stage half empty) in tiles of 16: a warp has two lanes.  96 groups, or 48 with two row blocks in one:
    # several per lane, of four giant steps; three keys and 25 inputs in 9 parts
    two_n = 2 << 10
    P, base = ckks.find_primes(1 << 60, two_n, 2)
    primes = [base if b == 60 else ckks.find_primes(1 << b, two_n, 8)[i] for i, b in enumerate(bits)]
    run_case(ckks.Params(1 << 10, primes, P, 2.0 ** 40), ckks.Plan(16, 1, 4, 4, **modes), 24 * 16 - 5, 25 * 16 - 3, 29, 1e-2,
             "tiles16", tight=1e-2)


def test_linear_gpt2_qkv_config_bit_exact():
    w = wl.WORKLOADS["gpt2_qkv"]
    par = oracle_params(w.params)
    L = w.layers[0]
    run_case(par, ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g), L.d_out, L.d_in, 0, 1e-3, L.name)


def check_blocks(par, plan, layers, blocks_of, seed, on_the_fly=(), splits=None):
    """Full-size calls exactly as the benchmark's runner issues them (projections that read the same
    activation stacked row-wise into one call, repeated on the same buffers so that the third call is the
    replayed graph with its concurrent key-switch chains): the device computes every output block, the
    oracle the listed ones; those must agree on every residue, before and after the rescale, and decrypt
    to the fp64 product.  Calls with the same d_in share one set of input ciphertexts, so that the
    oracle rotates them only once.  splits: {call name: (b, g)}, the calls whose weights are encoded with a
    baby/giant split of their own (as the runner does under the headline plan)."""
    splits = splits or {}
    assert not set(splits) & set(on_the_fly)        # the on-the-fly path runs under the plan's own split
    base = plan
    plans = {name: ckks.Plan(base.D, base.tau, b, g, base.pack, base.moddown, base.hoist) for name, (b, g) in splits.items()}
    extra = sorted({st for pl in plans.values() for st in ckks.required_rotations(pl)})
    s = ckks.keygen(par, seed)
    keys = ckks.make_rotation_keys(par, s, base, seed, extra_steps=extra)
    units = wl.fuse_shared_inputs(layers, base.D)
    inputs, rotated = {}, {}         # d_in -> (x, ciphertexts); (d_in, b) -> the oracle's baby rotations
    g = GpuSide(par, base)
    try:
        g.load_keys(keys, extra_steps=extra)
        for name, d_in, members in units:
            plan = plans.get(name, base)
            d_out = sum(m.d_out for m in members)
            W = np.concatenate([wl.gen_weights(seed, m.name, m.d_out, m.d_in) for m in members], axis=0)
            if d_in not in inputs:
                x = wl.gen_activation(seed, f"x{d_in}", d_in)
                inputs[d_in] = (x, ckks.encrypt_vector(par, base, s, x, seed))
            x, cts = inputs[d_in]
            if (d_in, plan.b) not in rotated:
                rot_fn = ckks.baby_rotations_ext if plan.hoist == "double" else ckks.baby_rotations
                rotated[(d_in, plan.b)] = [rot_fn(par, plan, ct, keys) for ct in cts]
            X = rotated[(d_in, plan.b)]
            n_in, n_out = len(cts), plan.n_out(d_out)
            blocks = list(blocks_of(name, n_out))
            expect = ckks.linear(par, plan, cts, W, keys, blocks=blocks, X=X)
            if name in splits:
                w = g.bf.bf_encode_weights_split(g.ctx, g.to_dev(W), d_out, d_in, plan.b, plan.g)
            else:
                w = g.bf.bf_encode_weights(g.ctx, g.to_dev(W), d_out, d_in)
            ct_in = g.to_dev(np.stack(cts))
            out = g.empty_u64(n_out, 2, par.r, par.N)
            for call in range(3):               # direct, captured, replayed
                out.zero_()
                g.bf.bf_linear(g.ctx, ct_in, n_in, w, None, d_out, d_in, out, n_out)
            if name in on_the_fly:          # the same call with the weights encoded on the fly
                fly = g.to_host_u64(g.linear(cts, W, d_out, d_in))
                for p in blocks:
                    assert np.array_equal(fly[p], expect[p]), (name, p, "on the fly")
                del fly
            low = g.empty_u64(n_out, 2, par.r - 1, par.N)
            scale = g.bf.bf_rescale(g.ctx, out, low, n_out, par.r, par.scale * par.scale)
            # the call the runner makes: product and rescale in one (direct, captured, replayed)
            low_fused = g.empty_u64(n_out, 2, par.r - 1, par.N)
            for call in range(3):
                low_fused.zero_()
                scale_fused = g.bf.bf_linear_rescaled(g.ctx, ct_in, n_in, w, None, d_out, d_in, low_fused, n_out,
                                                      par.scale * par.scale)
            assert scale_fused == scale
            got, low, low_fused = g.to_host_u64(out), g.to_host_u64(low), g.to_host_u64(low_fused)
            assert np.array_equal(low_fused, low), name       # every output ciphertext
            g.bf.bf_weights_free(g.ctx, w)
            y_ref = W.astype(np.float64) @ x
            for p in blocks:
                assert np.array_equal(got[p], expect[p]), (name, p)
                assert np.array_equal(low[p], ckks.rescale(par, expect[p])), (name, p)
                part = ckks.fold_output(ckks.decode(ckks.decrypt(par, s, low[p]), par.N, scale), plan, p, d_out)
                err = np.abs(part - y_ref[p * plan.rows_per_ct:p * plan.rows_per_ct + len(part)]).max()
                assert err < 1e-3, (name, p, err)
    finally:
        g.close()


@pytest.mark.parametrize("modes", [{}, BEST], ids=["plain", "best"])
def test_gpt2_step_one_whole_layer_every_block(modes):
    # config 2: one transformer layer of the GPT-2 decode step, all four calls, every output ciphertext
    # (qkv 3 row blocks, out_proj 1, ffn_up 3, ffn_down 1 with three input ciphertexts)
    w = wl.WORKLOADS["gpt2_step"]
    par = oracle_params(w.params)
    plan = ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g, **modes)
    check_blocks(par, plan, w.layers, lambda name, n_out: range(n_out), 11, splits=w.splits if modes else None)


@pytest.mark.parametrize("modes", [{}, BEST], ids=["plain", "best"])
def test_qwen3_step_the_calls_of_one_layer(modes):
    # config 3: the four calls the runner issues per layer.  q+k+v (1024 -> 4096) in full; o (2048 -> 1024, two
    # input ciphertexts) in full, also on the fly; gate+up (1024 -> 6144): its 18 giant rotations run as two
    # chains of 9 -- blocks 0 and 2 lie in the first chain for j = 1, 2 and in the second for j = 3, blocks 3
    # and 5 in the first for j = 1 and in the second for j = 2, 3; down (3072 -> 1024) in full.  With two row
    # blocks per ciphertext: every output ciphertext of every call
    w = wl.WORKLOADS["qwen3_step"]
    par = oracle_params(w.params)
    plan = ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g, **modes)
    pick = {"q+k+v": [0, 1, 2, 3], "o": [0], "gate+up": [0, 2, 3, 5], "down": [0]}
    blocks_of = (lambda name, n_out: range(n_out)) if modes else (lambda name, n_out: pick[name])
    check_blocks(par, plan, w.layers, blocks_of, 12, on_the_fly=("o",), splits=w.splits if modes else None)


@pytest.mark.parametrize("modes", [{}, BEST], ids=["plain", "best"])
def test_llama3_layer_the_calls_the_benchmark_times(modes):
    # config 4 at N = 2^16: q+k+v (4096 -> 6144): first block, the k block and the v block; o (4096 -> 4096):
    # first and last; gate+up (4096 -> 28672): 84 giant rotations in four launches of 22, 22, 22 and 18 --
    # rotation (j - 1) * 28 + p of block p, so block 0 meets launches 1, 2, 3; block 14 (first of up) 1, 2, 4;
    # blocks 21 and 22 the end of launch 1 and the start of launch 2; block 27 launches 2, 3 and the very last
    # rotation; down (14336 -> 4096): 14 input ciphertexts whose 98 baby rotations share two hoisted ModUps
    # (9 + 5 ciphertexts), every output block, and once more with the weights encoded on the fly.
    # With two row blocks per ciphertext gate+up has 14 outputs and 42 giant rotations in launches of 22 and 20:
    # rotation (j - 1) * 14 + p, so ciphertext 0 meets launch 1 twice and launch 2, ciphertexts 7 and 8 the end of
    # launch 1 and the start of launch 2, ciphertext 13 the very last rotation
    w = wl.WORKLOADS["llama3_layer"]
    par = oracle_params(w.params)
    plan = ckks.Plan(w.plan.D, w.plan.tau, w.plan.b, w.plan.g, **modes)
    if modes:
        pick = {"q+k+v": [0, 2], "o": [0, 1], "gate+up": [0, 7, 8, 13], "down": [0, 1]}
    else:
        pick = {"q+k+v": [0, 4, 5], "o": [0, 3], "gate+up": [0, 14, 21, 22, 27], "down": [0, 1, 2, 3]}
    # (under the headline plan gate+up and down run with splits of their own, 16 x 2 and 4 x 8; o is then the call
    # that is also checked with its weights encoded on the fly)
    check_blocks(par, plan, w.layers, lambda name, n_out: pick[name], 13, on_the_fly=("o",) if modes else ("down",),
                 splits=w.splits if modes else None)


def test_linear_with_the_papers_own_parameter_set():
    # N = 8192, primes of [60, 30, 30, 30] bits, scale 2^30, one 60-bit special prime (Sec. 4.2).  The 60-bit
    # ciphertext prime takes the whole-word accumulation paths of the multiply-accumulate and key-switch kernels.
    par = oracle_params("paper_n13")
    run_case(par, ckks.Plan(256, 16, 4, 4), 300, 520, 4, 1e-2, "paper_n13", tight=1e-3)   # scale 2^30: coarser


def test_repeated_calls_replay_a_graph_and_still_read_fresh_inputs():
    # from the third call with the same buffers on, bf_linear replays a captured launch sequence; the
    # data in those buffers may change between calls and results must follow
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4)
    s = ckks.keygen(par, 31)
    keys = ckks.make_rotation_keys(par, s, plan, 31)
    W = wl.gen_weights(31, "graph", 100, 130)
    xs = [wl.gen_activation(31, f"graph{t}", 130) for t in range(2)]
    cts = [ckks.encrypt_vector(par, plan, s, x, 31 + t) for t, x in enumerate(xs)]
    expect = [ckks.linear(par, plan, c, W, keys) for c in cts]
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        w = g.bf.bf_encode_weights(g.ctx, g.to_dev(W), 100, 130)
        ct_in = g.to_dev(np.stack(cts[0]))
        ct_out = g.empty_u64(2, 2, par.r, par.N)
        g.bf.bf_get_kernel_stats(g.ctx)            # reset the launch counters
        for call in range(6):
            which = call % 2
            ct_in.copy_(g.to_dev(np.stack(cts[which])))
            g.bf.bf_linear(g.ctx, ct_in, 3, w, None, 100, 130, ct_out, 2)
            got = g.to_host_u64(ct_out)
            for p in range(2):
                assert np.array_equal(got[p], expect[which][p]), (call, p)
        stats = g.bf.bf_get_kernel_stats(g.ctx)
        per_call = sum(v[0] for v in stats.values()) / 6
        assert per_call == int(per_call) and per_call > 5       # replays are counted like direct launches
        # turning replay off gives the same results
        g.bf.bf_set_graph_replay(g.ctx, False)
        g.bf.bf_linear(g.ctx, ct_in, 3, w, None, 100, 130, ct_out, 2)
        assert np.array_equal(g.to_host_u64(ct_out)[0], expect[1][0])
        # plain stream order instead of dependent launches, directly and replayed: same residues
        g.bf.bf_set_dependent_launch(g.ctx, False)
        g.bf.bf_set_graph_replay(g.ctx, True)
        for call in range(4):
            ct_out.zero_()
            g.bf.bf_linear(g.ctx, ct_in, 3, w, None, 100, 130, ct_out, 2)
            got = g.to_host_u64(ct_out)
            for p in range(2):
                assert np.array_equal(got[p], expect[1][p]), (call, p)
        # any number of concurrent key-switch chains, directly and replayed
        g.bf.bf_set_dependent_launch(g.ctx, True)
        for lanes in (1, 3, 4, 2):
            g.bf.bf_set_lanes(g.ctx, lanes)
            for call in range(3):
                ct_out.zero_()
                g.bf.bf_linear(g.ctx, ct_in, 3, w, None, 100, 130, ct_out, 2)
                got = g.to_host_u64(ct_out)
                for p in range(2):
                    assert np.array_equal(got[p], expect[1][p]), (lanes, call, p)
        # and the just-in-time encoding path under dependent launches
        for call in range(2):
            ct_out.zero_()
            g.bf.bf_linear(g.ctx, ct_in, 3, None, g.to_dev(W), 100, 130, ct_out, 2)
            got = g.to_host_u64(ct_out)
            for p in range(2):
                assert np.array_equal(got[p], expect[1][p]), (call, p)
    finally:
        g.close()


class _Device:
    """A context on the N = 2^15 ring with uniform keys, and a device with little memory left."""

    def __init__(self):
        import torch
        self.torch = torch
        self.par, self.plan = oracle_params("n15"), ckks.Plan(1024, 16, 16, 4)
        self.g = GpuSide(self.par, self.plan)
        self.bf, self.ctx, self.hog = self.g.bf, self.g.ctx, None

    def random_words(self, *shape):
        return self.torch.randint(0, min(self.par.basis), shape, dtype=self.torch.int64, device="cuda")

    def leave(self, nbytes):
        self.torch.cuda.synchronize()
        self.torch.cuda.empty_cache()
        self.hog = self.torch.empty(self.torch.cuda.mem_get_info()[0] - nbytes, dtype=self.torch.uint8, device="cuda")

    def close(self):
        self.hog = None
        self.torch.cuda.empty_cache()
        self.g.close()


def test_a_call_that_ran_out_of_memory_leaves_no_stale_launch_sequence():
    # a larger call gives up the scratch of a captured one before its own allocation fails: the next small call has to
    # allocate again, not replay a sequence that points into what was freed
    d = _Device()
    try:
        par, steps = d.par, list(ckks.required_rotations(d.plan))
        d.bf.bf_load_eval_keys(d.ctx, steps, len(steps), d.random_words(len(steps), par.r, 2, par.r + 1, par.N))
        small, large = (d.torch.randn(rows, 1024, device="cuda") * 0.02 for rows in (1024, 8192))
        ct, out, big = d.random_words(1, 2, par.r, par.N), d.g.empty_u64(1, 2, par.r, par.N), d.g.empty_u64(8, 2, par.r, par.N)
        w = d.bf.bf_encode_weights(d.ctx, small, 1024, 1024)
        call = lambda: d.bf.bf_linear(d.ctx, ct, 1, w, None, 1024, 1024, out, 1)
        for _ in range(3):
            call()
        expect = d.g.to_host_u64(out)
        d.leave(64 << 20)
        with pytest.raises(d.bf.BifrostError) as ei:
            d.bf.bf_linear(d.ctx, ct, 1, None, large, 8192, 1024, big, 8)
        assert ei.value.code == d.bf.BF_ERR_OOM
        for _ in range(3):
            out.zero_()
            call()
        assert np.array_equal(d.g.to_host_u64(out), expect)
    finally:
        d.close()


def test_encoding_needs_no_more_memory_than_small_passes_take():
    # 512 diagonals in one pass of the encoder would take 1.3 GB beside 0.64 GB of weights; in passes of 256 it is 0.67 GB
    d = _Device()
    try:
        W = d.torch.randn(8192, 1024, device="cuda") * 0.02
        expect, got = d.g.empty_u64(d.par.r, d.par.N), d.g.empty_u64(d.par.r, d.par.N)
        free = GpuSide(d.par, d.plan)               # (the same weights where memory is not short)
        try:
            w0 = free.bf.bf_encode_weights(free.ctx, W, 8192, 1024)
            picks = [(0, 0, 0, 0), (3, 0, 3, 15), (7, 0, 1, 2), (7, 0, 3, 15)]
            words = []
            for at in picks:
                free.bf.bf_weights_export(free.ctx, w0, *at, expect)
                words.append(free.to_host_u64(expect).copy())
        finally:
            free.close()
        d.torch.cuda.set_stream(d.g.stream)
        d.leave(1640 << 20)
        w = d.bf.bf_encode_weights(d.ctx, W, 8192, 1024)
        for at, want in zip(picks, words):
            d.bf.bf_weights_export(d.ctx, w, *at, got)
            assert np.array_equal(d.g.to_host_u64(got), want), at
    finally:
        d.close()


def test_unloading_keys_invalidates_replayed_launch_sequences():
    # after the keys are dropped, a call that was being replayed from its captured graph must be refused
    # (the graph holds the addresses of the freed key arrays), and reloading the keys must make it work again
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4)
    s = ckks.keygen(par, 51)
    keys = ckks.make_rotation_keys(par, s, plan, 51)
    W = wl.gen_weights(51, "unload", 100, 130)
    cts = ckks.encrypt_vector(par, plan, s, wl.gen_activation(51, "unload", 130), 51)
    expect = ckks.linear(par, plan, cts, W, keys)
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        w = g.bf.bf_encode_weights(g.ctx, g.to_dev(W), 100, 130)
        ct_in = g.to_dev(np.stack(cts))
        ct_out = g.empty_u64(2, 2, par.r, par.N)
        for call in range(4):                       # direct, captured, replayed, replayed
            g.bf.bf_linear(g.ctx, ct_in, 3, w, None, 100, 130, ct_out, 2)
        assert np.array_equal(g.to_host_u64(ct_out)[1], expect[1])
        g.bf.bf_get_kernel_stats(g.ctx)
        g.bf.bf_load_eval_keys(g.ctx, [], 0, None)
        with pytest.raises(g.bf.BifrostError) as ei:
            g.bf.bf_linear(g.ctx, ct_in, 3, w, None, 100, 130, ct_out, 2)
        assert ei.value.code == g.bf.BF_ERR_MISSING_KEY
        assert sum(v[0] for v in g.bf.bf_get_kernel_stats(g.ctx).values()) == 0     # nothing was launched
        g.load_keys(keys)
        for call in range(3):
            ct_out.zero_()
            g.bf.bf_linear(g.ctx, ct_in, 3, w, None, 100, 130, ct_out, 2)
        got = g.to_host_u64(ct_out)
        assert np.array_equal(got[0], expect[0]) and np.array_equal(got[1], expect[1])
    finally:
        g.close()


@pytest.mark.parametrize("modes", [{}, dict(moddown="per_output", hoist="double")], ids=["plain", "extended"])
@pytest.mark.parametrize("lanes", [3, 4])
def test_more_giant_rotations_than_one_launch_holds_with_three_and_four_lanes(lanes, modes):
    # 30 output blocks x 3 giant steps = 90 rotations: as one chain they go in launches of lanes * floor(64 / lanes)
    # rotations, which must not exceed the 64 a launch holds (with 3 lanes: 63); also with the inner sums kept in the
    # extended basis (30 outputs assembled from 90 key-switch results)
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4, **modes)
    d_out, d_in = 1920, 64
    s = ckks.keygen(par, 52)
    keys = ckks.make_rotation_keys(par, s, plan, 52)
    W = wl.gen_weights(52, "lanes", d_out, d_in)
    cts = ckks.encrypt_vector(par, plan, s, wl.gen_activation(52, "lanes", d_in), 52)
    blocks = [0, 20, 21, 29]
    expect = ckks.linear(par, plan, cts, W, keys, blocks=blocks)
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        g.bf.bf_set_lanes(g.ctx, lanes)
        w = g.bf.bf_encode_weights(g.ctx, g.to_dev(W), d_out, d_in)
        ct_in = g.to_dev(np.stack(cts))
        ct_out = g.empty_u64(30, 2, par.r, par.N)
        for call in range(3):                       # direct, captured, replayed
            ct_out.zero_()
            g.bf.bf_linear(g.ctx, ct_in, 1, w, None, d_out, d_in, ct_out, 30)
            got = g.to_host_u64(ct_out)
            for p in blocks:
                assert np.array_equal(got[p], expect[p]), (call, p)
    finally:
        g.close()


@pytest.mark.parametrize("pkey,plan_t,shape", [
    ("n12", (64, 4, 4, 4), (100, 130)),          # tau = 4: rotations by 1 and 2, two output ciphertexts
    ("n12", (32, 32, 1, 1), (70, 50)),           # tau = 32, no other rotation in the plan, three outputs
    ("n15", (1024, 16, 16, 4), (1100, 300)),     # the headline plan: rotations by 1, 2, 4, 8
])
def test_fold_in_ciphertext_matches_oracle(pkey, plan_t, shape):
    par = oracle_params(pkey)
    plan = ckks.Plan(*plan_t)
    d_out, d_in = shape
    s = ckks.keygen(par, 41)
    fold_steps = ckks.fold_rotations(plan)
    keys = ckks.make_rotation_keys(par, s, plan, 41, extra_steps=fold_steps)
    W = wl.gen_weights(41, "fold", d_out, d_in)
    x = wl.gen_activation(41, "fold", d_in)
    cts = ckks.encrypt_vector(par, plan, s, x, 41)
    n_out = -(-d_out // plan.D)
    lin = ckks.linear(par, plan, cts, W, keys)
    expect = [ckks.fold_in_ciphertext(par, plan, lin[p], keys) for p in range(n_out)]
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys, extra_steps=fold_steps)
        out = g.linear(cts, W, d_out, d_in, weights=g.bf.bf_encode_weights(g.ctx, g.to_dev(W), d_out, d_in))
        g.bf.bf_fold(g.ctx, out, n_out)
        got = g.to_host_u64(out)
        for p in range(n_out):
            assert np.array_equal(got[p], expect[p]), p
        # rescale, decrypt: slot (0, kappa, 0) is the complete dot product
        low = g.empty_u64(n_out, 2, par.r - 1, par.N)
        scale = g.bf.bf_rescale(g.ctx, out, low, n_out, par.r, par.scale * par.scale)
        low = g.to_host_u64(low)
        y = np.zeros(d_out)
        for p in range(n_out):
            part = ckks.folded_output(ckks.decode(ckks.decrypt(par, s, low[p]), par.N, scale), plan, p, d_out)
            y[p * plan.D:p * plan.D + len(part)] = part
        assert np.abs(y - W.astype(np.float64) @ x).max() < 1e-3
        # without the keys of the fold the call is refused before anything is launched
        g2 = GpuSide(par, plan)
        try:
            g2.load_keys(keys)
            if fold_steps and not set(fold_steps) <= set(ckks.required_rotations(plan)):
                with pytest.raises(g2.bf.BifrostError) as ei:
                    g2.bf.bf_fold(g2.ctx, out, n_out)
                assert ei.value.code == g2.bf.BF_ERR_MISSING_KEY
        finally:
            g2.close()
    finally:
        g.close()


@pytest.mark.parametrize("pkey", ["n12", "paper_n13"])        # ciphertext primes below 2^50, and one of 60 bits
@pytest.mark.parametrize("tau", [2, 8])                       # one round (which ends in the other buffer), an odd number of them
def test_fold_rounds_and_rotation_in_place(pkey, tau):
    par = oracle_params(pkey)
    plan = ckks.Plan(8 * tau, tau, 4, 2)
    s = ckks.keygen(par, 47)
    keys = ckks.make_rotation_keys(par, s, plan, 47, extra_steps=ckks.fold_rotations(plan))
    cts = np.stack([np.ascontiguousarray(wl.gen_uniform_residues(47, f"fold{t}", par.primes, (2, par.N)).transpose(1, 0, 2))
                    for t in range(3)])
    g = GpuSide(par, plan)
    try:
        steps = g.load_keys(keys, extra_steps=ckks.fold_rotations(plan))
        d = g.to_dev(cts)
        g.bf.bf_fold(g.ctx, d, len(cts))
        got = g.to_host_u64(d)
        for t in range(len(cts)):
            assert np.array_equal(got[t], ckks.fold_in_ciphertext(par, plan, cts[t], keys)), t
        d = g.to_dev(cts[0])
        g.bf.bf_rotate(g.ctx, d, steps[-1], d)
        assert np.array_equal(g.to_host_u64(d), ckks.rotate(par, cts[0], steps[-1], keys))
    finally:
        g.close()


def test_fold_of_more_ciphertexts_than_one_key_switch_batch():
    # 70 ciphertexts: the rounds run in two batches (64 + 6); sampled ones are compared with the oracle
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4)
    s = ckks.keygen(par, 43)
    fold_steps = ckks.fold_rotations(plan)
    keys = ckks.make_rotation_keys(par, s, plan, 43, extra_steps=fold_steps)
    n_ct = 70
    # [r][2][N] uniform residues per ciphertext, rearranged to the boundary layout [2][r][N]
    cts = np.stack([np.ascontiguousarray(wl.gen_uniform_residues(43, f"fold{t}", par.primes, (2, par.N)).transpose(1, 0, 2))
                    for t in range(n_ct)])
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys, extra_steps=fold_steps)
        d = g.to_dev(cts)
        g.bf.bf_fold(g.ctx, d, n_ct)
        got = g.to_host_u64(d)
        for t in (0, 1, 63, 64, 69):
            assert np.array_equal(got[t], ckks.fold_in_ciphertext(par, plan, cts[t], keys)), t
    finally:
        g.close()


@pytest.mark.parametrize("n_primes,n_ct", [
    (2, 55),        # 16 chunks of a ring of 2^12, two digits: four chunks a block
    (2, 27),        # ... two, so that the launch fills the GPU
    (4, 16),        # four digits, two chunks: all eight warps
])
def test_fold_with_several_chunks_in_a_block(n_primes, n_ct):
    par = ckks.Params(1 << 12, ckks.find_primes(1 << 40, 2 << 12, n_primes), ckks.find_primes(1 << 60, 2 << 12, 1)[0], 2.0 ** 30)
    plan = ckks.Plan(4, 2, 2, 1)
    s = ckks.keygen(par, 53)
    keys = ckks.make_rotation_keys(par, s, plan, 53, extra_steps=ckks.fold_rotations(plan))
    cts = np.stack([np.ascontiguousarray(wl.gen_uniform_residues(53, f"fold{t}", par.primes, (2, par.N)).transpose(1, 0, 2))
                    for t in range(n_ct)])
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys, extra_steps=ckks.fold_rotations(plan))
        d = g.to_dev(cts)
        g.bf.bf_fold(g.ctx, d, n_ct)
        got = g.to_host_u64(d)
        for t in (0, 1, n_ct // 2, n_ct - 1):
            assert np.array_equal(got[t], ckks.fold_in_ciphertext(par, plan, cts[t], keys)), t
    finally:
        g.close()


@pytest.mark.parametrize("modes", [{}, BEST], ids=["plain", "best"])
def test_fallback_path_in_several_rounds_of_its_scratch(modes):
    # the on-the-fly path encodes output groups in rounds bounded by a scratch size: one group per round,
    # two per round with a ragged last round, and everything in one round must give the oracle's residues
    # (headline plan: rounds that start in the middle of a giant step, whose rotated parts are stored permuted)
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4, **modes)
    d_out, d_in = 150, 130                        # 3 output blocks x 4 giant steps = 12 groups of 3 x 4 terms
    s = ckks.keygen(par, 31)
    keys = ckks.make_rotation_keys(par, s, plan, 31)
    W = wl.gen_weights(31, "rounds", d_out, d_in)
    x = wl.gen_activation(31, "rounds", d_in)
    cts = ckks.encrypt_vector(par, plan, s, x, 31)
    expect = ckks.linear(par, plan, cts, W, keys)
    group_bytes = 3 * 4 * (par.r + (1 if modes else 0)) * par.N * 8
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        for bound in (1, 5 * group_bytes + 17, 2 * group_bytes, 3 * group_bytes, 1 << 32):
            g.bf.bf_set_encode_scratch(g.ctx, bound)
            got = g.to_host_u64(g.linear(cts, W, d_out, d_in))
            for p in range(plan.n_out(d_out)):
                assert np.array_equal(got[p], expect[p]), (bound, p)
        with pytest.raises(g.bf.BifrostError):
            g.bf.bf_set_encode_scratch(g.ctx, 0)
    finally:
        g.close()


def test_stacking_projections_that_share_an_input_changes_no_residue():
    # q/k/v (or gate/up) read the same activation: one call over the row-stacked matrix must give
    # exactly the ciphertexts of the separate calls
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4)
    s = ckks.keygen(par, 21)
    keys = ckks.make_rotation_keys(par, s, plan, 21)
    x = wl.gen_activation(21, "shared", 100)
    cts = ckks.encrypt_vector(par, plan, s, x, 21)
    W1 = wl.gen_weights(21, "w1", 128, 100)
    W2 = wl.gen_weights(21, "w2", 64, 100)
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        o1 = g.to_host_u64(g.linear(cts, W1, 128, 100))
        o2 = g.to_host_u64(g.linear(cts, W2, 64, 100))
        both = g.to_host_u64(g.linear(cts, np.concatenate([W1, W2]), 192, 100))
        assert np.array_equal(both[:2], o1) and np.array_equal(both[2:], o2)
        expect = ckks.linear(par, plan, cts, W2, keys)
        assert np.array_equal(o2[0], expect[0])
    finally:
        g.close()


def test_structured_matrices_on_device():
    par = oracle_params("n12")
    plan = ckks.Plan(64, 4, 4, 4)
    s = ckks.keygen(par, 5)
    keys = ckks.make_rotation_keys(par, s, plan, 5)
    x = wl.gen_activation(5, "struct", 64)
    cts = ckks.encrypt_vector(par, plan, s, x, 5)
    g = GpuSide(par, plan)
    try:
        g.load_keys(keys)
        mats = {"zero": np.zeros((64, 64), np.float32), "identity": np.eye(64, dtype=np.float32),
                "shift": np.roll(np.eye(64, dtype=np.float32), 5, axis=1)}
        single = np.zeros((64, 64), np.float32)
        single[17, 42] = 1.5
        mats["single"] = single
        for name, W in mats.items():
            got = g.to_host_u64(g.linear(cts, W, 64, 64))
            low = ckks.rescale(par, got[0])
            scale = par.scale * par.scale / par.primes[-1]
            y = ckks.fold_output(ckks.decode(ckks.decrypt(par, s, low), par.N, scale), plan, 0, 64)
            assert np.abs(y - W.astype(np.float64) @ x).max() < 1e-6, name
    finally:
        g.close()


def test_error_paths_do_not_touch_the_device():
    import torch
    from paper_2606_17421_b200 import bifrost as bf
    ps = wl.PARAM_SETS["n12"]
    plan = bf.bf_plan(64, 1, 8, 8)
    basis = list(ps["primes"]) + [ps["special"]]
    with pytest.raises(bf.BifrostError) as ei:
        bf.bf_ctx_create(ps["N"], basis[:-1] + [basis[0]], 3, 2.0 ** 40, plan)      # duplicate prime
    assert ei.value.code == bf.BF_ERR_BAD_PRIME
    with pytest.raises(bf.BifrostError) as ei:
        bf.bf_ctx_create(ps["N"], [basis[0] + 2] + basis[1:], 3, 2.0 ** 40, plan)   # not 1 mod 2N
    assert ei.value.code == bf.BF_ERR_BAD_PRIME
    with pytest.raises(bf.BifrostError) as ei:
        bf.bf_ctx_create(ps["N"], basis, 3, 2.0 ** 40, bf.bf_plan(64, 1, 8, 4))
    assert ei.value.code == bf.BF_ERR_SHAPE
    with pytest.raises(bf.BifrostError) as ei:
        bf.bf_ctx_create(3000, basis, 3, 2.0 ** 40, plan)
    assert ei.value.code == bf.BF_ERR_INVALID_ARG
    ctx = bf.bf_ctx_create(ps["N"], basis, 3, 2.0 ** 40, plan)
    try:
        ct = torch.zeros((1, 2, 3, ps["N"]), dtype=torch.int64, device="cuda")
        W = torch.zeros((64, 64), dtype=torch.float32, device="cuda")
        with pytest.raises(bf.BifrostError) as ei:          # no keys loaded
            bf.bf_linear(ctx, ct, 1, None, W, 64, 64, ct.clone(), 1)
        assert ei.value.code == bf.BF_ERR_MISSING_KEY
        with pytest.raises(bf.BifrostError) as ei:          # wrong number of input ciphertexts
            bf.bf_linear(ctx, ct, 2, None, W, 64, 64, ct.clone(), 1)
        assert ei.value.code == bf.BF_ERR_SHAPE
        low = torch.zeros((1, 2, 2, ps["N"]), dtype=torch.int64, device="cuda")
        with pytest.raises(bf.BifrostError) as ei:          # the fused call reports the same errors
            bf.bf_linear_rescaled(ctx, ct, 1, None, W, 64, 64, low, 1)
        assert ei.value.code == bf.BF_ERR_MISSING_KEY
        with pytest.raises(bf.BifrostError) as ei:
            bf.bf_linear_rescaled(ctx, ct, 2, None, W, 64, 64, low, 1)
        assert ei.value.code == bf.BF_ERR_SHAPE
        with pytest.raises(bf.BifrostError) as ei:          # no output buffer
            bf.bf_linear_rescaled(ctx, ct, 1, None, W, 64, 64, None, 1)
        assert ei.value.code == bf.BF_ERR_INVALID_ARG
        bf.bf_set_cache_budget(ctx, 1000)
        with pytest.raises(bf.BifrostError) as ei:
            bf.bf_encode_weights(ctx, W, 64, 64)
        assert ei.value.code == bf.BF_ERR_OOM
        with pytest.raises(bf.BifrostError) as ei:          # (the budget is checked after the split)
            bf.bf_encode_weights_split(ctx, W, 64, 64, 16, 4)
        assert ei.value.code == bf.BF_ERR_OOM
        with pytest.raises(bf.BifrostError) as ei:
            bf.bf_encode_weights_split(ctx, W, 64, 64, 16, 8)
        assert ei.value.code == bf.BF_ERR_SHAPE
    finally:
        bf.bf_ctx_destroy(ctx)
