"""Edges of the GPU kernels' tiles and ranges against the oracle: clusters and super-clusters of the
pair histograms, chunks, layouts and molecule sizes of the sweep, node grids of the smeared
histogram, and the two places the fit keeps its columns in.

Bars as in test_gpu_parity: counts and coordinates exact, dU within 1e-5 of its condition scale plus
1e-4 kJ/mol; those of the smeared form and of the fit are derived where they stand.
"""
import numpy as np
import pytest

import oracle
from paper_1904_08756_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1904_08756_gb300 import epsr  # noqa: E402
from test_gpu_parity import DEV, gpu_hist, replay, run_logged  # noqa: E402


def mixed_box(sizes, n_mol, n_types, seed, n_bins=200, spacing=4.0, r_lj=0.0):
    """Rigid molecules of the sizes given in turn, on a jittered cubic lattice; types at random, every
    other type without a Lennard-Jones term, charges +-0.3 e."""
    rng = np.random.default_rng(seed)
    k = int(np.ceil(n_mol ** (1 / 3) - 1e-9))
    L_fx = int(synth.SCALE * spacing * max(k, 4))
    at = rng.permutation(k ** 3)[:n_mol]
    centre = (np.stack([at % k, at // k % k, at // (k * k)], 1) + 0.5) * spacing
    m = np.array([sizes[i % len(sizes)] for i in range(n_mol)])
    start = np.concatenate([[0], np.cumsum(m)])
    off = rng.normal(size=(start[-1], 3))
    off *= 0.9 / np.linalg.norm(off, axis=1, keepdims=True)
    off[start[:-1][m == 1]] = 0.0
    xyz = (np.repeat(centre, m, axis=0) + off + rng.uniform(-0.3, 0.3, (n_mol, 3)).repeat(m, axis=0)) * synth.SCALE
    return synth.System(name="mixed", L_fx=L_fx, xyz=(np.rint(xyz).astype(np.int64) % L_fx).astype(np.int32),
                        type=rng.integers(0, n_types, start[-1]).astype(np.int32), mol_start=start.astype(np.int64),
                        type_names=[f"T{i}" for i in range(n_types)], q=[0.3 - 0.6 * (i % 2) for i in range(n_types)],
                        sigma=[2.0 + 0.1 * i for i in range(n_types)], eps=[0.4 * (i % 2 == 0) for i in range(n_types)],
                        b=[5.0] * n_types, r_coul=7.0, bin_p=1, bin_q=25, n_bins=n_bins, rigid_molecules=max(sizes) > 1,
                        Q=0.5 + np.arange(50) * 0.1, r_lj=r_lj, seed=seed)


@pytest.mark.parametrize("n,L,types,bins", [(31, 30.0, 1, 150), (32, 30.0, 2, 150), (33, 30.0, 2, 150),
                                            (1024, 30.0, 3, 150), (1056, 30.0, 8, 150), (4097, 50.0, 2, 150),
                                            (4097, 50.0, 1, 800), (300, 2000.0, 2, 4000), (1100, 30.0, 8, 800)])
def test_cluster_histogram_edges(n, L, types, bins):
    """Full and partial clusters and super-clusters; ranges below and above half the box; clusters too
    wide for relative coordinates (a sparse box of 2,000 A); rows that leave no room in shared memory."""
    s = synth.uniform_gas(n, L, seed=n + types, n_types=types)
    s.bin_p, s.bin_q, s.n_bins = 1, 25, bins
    H = gpu_hist(epsr.Box(s)).reshape(-1, bins)
    assert np.array_equal(H, oracle.Box(s).histogram(threads=8))


@pytest.mark.parametrize("sizes,n_mol,types,bins,ctas,r_lj,ep", [
    ([3], 1, 2, 100, 0, 0.0, False),                       # one molecule: every batch is one move
    ([1], 33, 1, 100, 0, 0.0, True),                       # two chunks, the second with one atom
    ([2, 3], 300, 3, 100, 7, 0.0, True),                   # batches of 32, unaligned gather rows
    (list(range(1, 9)), 300, 8, 100, 0, 0.0, True),        # every molecule size and type
    (list(range(1, 9)), 300, 5, 100, 9, 6.0, True),        # the same with Lennard-Jones cut
    ([1, 4], 400, 4, 2000, 0, 0.0, True),                  # 80 KB of tables in shared memory
    ([1, 2], 4000, 8, 640, 1, 0.0, True),                  # 92 KB of tables, slices in global memory
], ids=["one", "chunk-end", "groups", "sizes", "sizes-cut", "tables", "tables-global"])
def test_sweep_edges_replay(sizes, n_mol, types, bins, ctas, r_lj, ep):
    s = mixed_box(sizes, n_mol, types, seed=n_mol + types, n_bins=bins, r_lj=r_lj)
    P = types * (types + 1) // 2
    table = (np.random.default_rng(5).normal(size=(P, bins)) * 0.3).astype(np.float32) if ep else None
    box = epsr.Box(s)
    if ep:
        box.epsr_box_set_ep(0, table)
    if ctas:
        box.epsr_mc_set_ctas(ctas)
    stats, log = run_logged(box, 600, seed=8)
    ob, _, _, flips = replay(s, s.xyz, log[0], 8, ep=table.astype(np.float64) if ep else None)
    assert flips <= 2
    assert np.array_equal(box.epsr_box_get_coords(), ob.xyz)


@pytest.mark.parametrize("n,L,sigma,bin_q", [(33, 20.0, 0.05, 25), (1057, 22.0, 0.02, 25), (1057, 40.0, 0.3, 5),
                                             (1057, 40.0, 0.05, 5), (65, 300.0, 0.05, 25)],
                         ids=["one-atom-cluster", "fine-nodes", "wide", "direct", "sparse"])
def test_smeared_edges(n, L, sigma, bin_q):
    """Histogram within 1e-5 of its largest entry (the rounding of the 2^-20 weights and of FP32
    distances), gradient of a smooth functional within 1e-4 in the 2-norm, as in test_gpu_parity."""
    s = synth.uniform_gas(n, L, seed=n, n_types=2)
    s.bin_p, s.bin_q, s.n_bins = 1, bin_q, 8 * bin_q
    box, ob = epsr.Box(s), oracle.Box(s)
    Ht = torch.zeros(box.hist_len, dtype=torch.float64, device=DEV)
    box.epsr_gr_smeared_fwd(sigma, Ht)
    ref = ob.smeared_hist(sigma)
    assert np.abs(Ht.cpu().numpy().reshape(ref.shape) - ref).max() <= 1e-5 * np.abs(ref).max()
    lam = np.cos(np.arange(3 * s.n_bins).reshape(3, -1) * s.dr * 2.0)
    _, factor = oracle.smeared_g(ob, ref)                              # g = Ht factor
    grad = torch.zeros((n, 3), dtype=torch.float32, device=DEV)
    box.epsr_gr_smeared_bwd(sigma, torch.from_numpy((lam / factor).astype(np.float32).reshape(-1)).to(DEV), grad)
    gref = ob.smeared_grad(sigma, lam)
    assert np.linalg.norm(grad.cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref)


def test_smeared_moments_do_not_wrap():
    """40,000 atoms on two points: all 4e8 pairs that are apart fall on one node, hundreds of times what
    a 32-bit moment holds. The offset from the node is rounded to 2^-13 (4e-7 A) and the distance of 2 A to 2e-7 A for
    every pair alike; the steepest weight changes by 2.9 per A and the largest is 0.24: 8e-6 of it."""
    n = 40000
    s = synth.uniform_gas(n, 30.0, seed=1, n_types=1)
    s.bin_p, s.bin_q, s.n_bins = 3, 100, 100
    s.xyz[:] = int(5 * synth.SCALE)
    s.xyz[n // 2:, 0] += int(2 * synth.SCALE) + 12345
    box = epsr.Box(s)
    Ht = torch.zeros(box.hist_len, dtype=torch.float64, device=DEV)
    box.epsr_gr_smeared_fwd(0.05, Ht)
    two = synth.System(**{**s.__dict__, "xyz": s.xyz[[0, n - 1]].copy(), "type": s.type[:2], "mol_start": s.mol_start[:3]})
    ref = oracle.Box(two).smeared_hist(0.05)[0] * (n // 2) ** 2
    assert np.abs(Ht.cpu().numpy() - ref).max() <= 2e-5 * ref.max()


@pytest.mark.parametrize("nQ,n_basis", [(6, 6), (13, 5), (999, 24), (20000, 20)],
                         ids=["square", "few-rows", "uneven-rows", "columns-in-global-memory"])
def test_ep_fit_edges(nQ, n_basis):
    """The fitted Delta S within 1e-8 of its largest (the bar of test_gpu_parity); rows fewer than the
    CTAs' shares, as many as the functions, and more than shared memory holds."""
    s = synth.water_box(60, seed=3, L_A=14.0)
    box = epsr.Box(s)
    rng = np.random.default_rng(nQ)
    Q = np.linspace(0.4, 25.0, nQ)
    w = rng.uniform(0.05, 0.3, (3, 3))
    F = oracle.ep_basis_matrix(n_basis, 0.5, Q.astype(np.float32).astype(np.float64), s.n_atoms / s.L ** 3)
    dS = (w @ (rng.normal(size=(3, n_basis)) * 0.01 @ F.T)).astype(np.float32)
    C = box.epsr_ep_update(0, torch.from_numpy(dS).to(DEV), w, Q, n_basis=n_basis, s_basis=0.5, gamma=0.0, alpha=1.0)
    dSp = oracle.pair_resolve(dS.astype(np.float64), w, 0.0)
    assert np.abs(C @ F.T - oracle.ep_fit(dSp, F) @ F.T).max() <= 1e-8 * np.abs(dSp).max()


def test_smeared_forward_repeats():
    """Partners up to about 20 A from an i-cluster's centre, where relative coordinates are rounded: the
    sums are the same bits in every call (the order of the clusters may not depend on timing)."""
    s = synth.uniform_gas(30000, 76.8, seed=9, n_types=2)
    s.bin_p, s.bin_q, s.n_bins = 1, 25, 350
    box = epsr.Box(s)
    Ht = torch.zeros((8, box.hist_len), dtype=torch.float64, device=DEV)
    for row in Ht:
        box.epsr_gr_smeared_fwd(0.05, row)
    assert torch.equal(Ht[0].expand_as(Ht), Ht)


@pytest.mark.parametrize("types", [(2, 1, 3), (4, 2, 5)], ids=["nodes", "direct"])
def test_smeared_boxes_of_one_handle(types):
    """Boxes of different types, sizes and bins in one handle, each against the oracle with the bars of
    test_smeared_edges; on the node grid, and with more types than it holds, pair by pair from queues."""
    systems = []
    for i, (n, L, bins) in enumerate([(2100, 27.0, 200), (40, 20.0, 160), (1057, 22.0, 120)]):
        s = synth.uniform_gas(n, L, seed=n, n_types=types[i])
        s.bin_p, s.bin_q, s.n_bins = 1, 25, bins
        systems.append(s)
    box = epsr.Box(systems)
    Ht = torch.zeros(box.hist_len, dtype=torch.float64, device=DEV)
    box.epsr_gr_smeared_fwd(0.05, Ht)
    dgt, want = [], []
    h0 = 0
    for s in systems:
        ob = oracle.Box(s)
        ref = ob.smeared_hist(0.05)
        got = Ht[h0:h0 + ref.size].cpu().numpy().reshape(ref.shape)
        assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
        h0 += ref.size
        lam = np.cos(np.arange(ref.size).reshape(ref.shape) * s.dr * 2.0)
        _, factor = oracle.smeared_g(ob, ref)
        dgt.append((lam / factor).astype(np.float32).reshape(-1))
        want.append(ob.smeared_grad(0.05, lam))
    grad = torch.zeros((box.n_atoms, 3), dtype=torch.float32, device=DEV)
    box.epsr_gr_smeared_bwd(0.05, torch.from_numpy(np.concatenate(dgt)).to(DEV), grad)
    a0 = 0
    for g in want:
        assert np.linalg.norm(grad[a0:a0 + len(g)].cpu().numpy() - g) <= 1e-4 * np.linalg.norm(g)
        a0 += len(g)


def test_smeared_handles_of_many_boxes():
    """A handle of 1,000 boxes holds no workspace of its own per box (it was 0.7 MB each); 400 boxes that
    need more than the workspace are taken in groups: boxes at the groups' ends against the oracle with
    the bars of test_smeared_edges."""
    s = synth.uniform_gas(30, 20.0, seed=2, n_types=2)
    s.bin_p, s.bin_q, s.n_bins = 1, 25, 200
    free, held = [], []
    for n in (100, 1000):
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
        held.append(epsr.Box([s] * n))
    free.append(torch.cuda.mem_get_info()[0])
    assert (free[1] - free[2]) - (free[0] - free[1]) < 200 << 20
    for h in held:
        h.close()
    systems = []
    for i in range(400):
        s = synth.uniform_gas(900, 16.0, seed=i, n_types=2)
        s.bin_p, s.bin_q, s.n_bins = 1, 25, 200
        systems.append(s)
    box = epsr.Box(systems)
    Ht = torch.zeros(box.hist_len, dtype=torch.float64, device=DEV)
    box.epsr_gr_smeared_fwd(0.05, Ht)
    lam = np.cos(np.arange(600).reshape(3, -1) * 0.08)
    ob = oracle.Box(systems[0])
    _, factor = oracle.smeared_g(ob, ob.smeared_hist(0.05))
    dgt = np.tile((lam / factor).astype(np.float32).reshape(-1), 400)
    grad = torch.zeros((box.n_atoms, 3), dtype=torch.float32, device=DEV)
    box.epsr_gr_smeared_bwd(0.05, torch.from_numpy(dgt).to(DEV), grad)
    for b in [0, 1, *range(325, 333), 399]:
        ob = oracle.Box(systems[b])
        ref, gref = ob.smeared_hist(0.05), ob.smeared_grad(0.05, lam)
        assert np.abs(Ht[600 * b:600 * b + 600].cpu().numpy().reshape(3, -1) - ref).max() <= 1e-5 * np.abs(ref).max()
        assert np.linalg.norm(grad[900 * b:900 * b + 900].cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref)


@pytest.mark.parametrize("n,L,boxes", [(60, 10.0, 300), (2, 9.0, 200)], ids=["few-pairs", "two-atoms"])
def test_smeared_many_small_boxes(n, L, boxes):
    """Handles of many boxes with few pairs each, which are smeared pair by pair: every box against the
    oracle with the bars of test_smeared_edges (and one weight's rounding, 2^-21, for single pairs)."""
    systems = []
    for i in range(boxes):
        s = synth.uniform_gas(n, L, seed=1000 + i, n_types=2)
        s.bin_p, s.bin_q, s.n_bins = 3, 100, 140 + i % 3
        systems.append(s)
    box = epsr.Box(systems)
    Ht = torch.zeros(box.hist_len, dtype=torch.float64, device=DEV)
    box.epsr_gr_smeared_fwd(0.05, Ht)
    h0 = 0
    for s in systems:
        ref = oracle.Box(s).smeared_hist(0.05)
        got = Ht[h0:h0 + ref.size].cpu().numpy().reshape(ref.shape)
        assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max() + 2.0 ** -21
        h0 += ref.size


def test_energy_change_error_with_many_ctas():
    """The error of dU may not grow with the CTAs a box is spread over: 9,999-atom water with a smooth
    empirical potential on 152 CTAs. In the 2-norm over the moves, plain FP32 sums of the partials have
    1.05e-7 of dU on a box of this kind, compensated ones 0.84e-7 (both known to 2 % from 3,000 moves);
    the bar is between the two."""
    s = synth.water_box(3333, seed=17)
    r = (np.arange(s.n_bins) + 0.5) * s.dr
    rng = np.random.default_rng(18)
    amp, k, ph = rng.uniform(0.1, 0.4, (3, 1)), rng.uniform(1.0, 2.5, (3, 1)), rng.uniform(0, 6.28, (3, 1))
    ep = (amp * np.cos(k * r + ph) * np.exp(-r / 4.0)).astype(np.float32)
    box = epsr.Box(s)
    box.epsr_box_set_ep(0, ep)
    _, log = run_logged(box, 3000, seed=19)
    ob = oracle.Box(s, ep=ep.astype(np.float64))
    err = ref = 0.0
    for t, e in enumerate(log[0]):
        mol, trial, _ = ob.propose(19, t, 0)
        dU, _ = ob.delta_u(mol, trial)
        err += (float(e["dU"]) - dU) ** 2
        ref += dU ** 2
        if e["accepted"]:
            ob.apply(mol, trial)
    assert np.sqrt(err / ref) <= 0.95e-7


def test_rotation_of_a_wide_molecule():
    """Trial coordinates of a molecule whose atoms lie 690 A to both sides of the first (three times the
    offset is past 2^31 grid units), wherever the rotated sum fits 32 bits again."""
    s = synth.uniform_gas(3, 100.0, seed=1, n_types=1)
    s.L_fx, s.mol_start, s.rigid_molecules = 2147483646, np.array([0, 3]), True
    s.max_translation, s.max_rotation_deg = 0.0, 60.0
    s.xyz = np.array([[5, 6, 7], [25, 6, 7], [5, 9, 7]], np.int32)
    box = epsr.Box(s)
    a = 720000000
    wide = np.array([[1000000000, 5, 3], [1000000000 + a, 5, 3], [1000000000 - a, 5, 3]], np.int32)
    checked = 0
    for t in range(40):
        box.epsr_box_set_coords(wide)
        _, log = run_logged(box, 1, seed=3, move0=t)
        _, trial, _ = oracle.Box(s, xyz=wide).propose(3, t)
        p = (trial.astype(np.int64) - wide[0] + s.L_fx // 2) % s.L_fx - s.L_fx // 2
        if (np.abs(p) * 3 + 3 < 2 ** 31).all():
            checked += 1
            assert np.array_equal(log[0][0]["trial"][:3], trial)
    assert checked > 20


def test_sweep_small_boxes_replay():
    """Boxes around the size up to which one CTA sweeps alone (and prepares a batch after the decisions of the
    one before), in one handle: every move of every box against the oracle."""
    systems = [mixed_box([1], 12, 2, seed=1), mixed_box([1, 3], 32, 3, seed=2), mixed_box([1], 65, 2, seed=3),
               mixed_box([3], 2, 2, seed=4), mixed_box([1, 2], 140, 2, seed=5)]
    box = epsr.Box(systems)
    _, log = run_logged(box, 500, seed=21)
    xyz = box.epsr_box_get_coords()
    a0 = 0
    for b, s in enumerate(systems):
        ob, _, _, flips = replay(s, s.xyz, log[b], 21, box_index=b)
        assert flips <= 2
        assert np.array_equal(xyz[a0:a0 + s.n_atoms], ob.xyz)
        a0 += s.n_atoms


@pytest.mark.parametrize("types,bins,n", [(8, 848, 60), (7, 1080, 60), (6, 1440, 40), (8, 700, 3000)])
def test_sweep_largest_tables_replay(types, bins, n):
    """The largest empirical potentials that boxes were made with (122 KB at 8 types), in small boxes and with
    slices in global memory: every move against the oracle."""
    s = mixed_box([1], n, types, seed=types, n_bins=bins)
    P = types * (types + 1) // 2
    table = (np.random.default_rng(6).normal(size=(P, bins)) * 0.3).astype(np.float32)
    box = epsr.Box(s)
    box.epsr_box_set_ep(0, table)
    _, log = run_logged(box, 400, seed=22)
    ob, _, _, flips = replay(s, s.xyz, log[0], 22, ep=table.astype(np.float64))
    assert flips <= 2
    assert np.array_equal(box.epsr_box_get_coords(), ob.xyz)


def test_histogram_of_a_mixed_handle():
    """Both histogram entries on boxes of 900 to 12,000 atoms of one to three types, against the all-pairs kernel
    over every tile and, box by box, the oracle."""
    systems = [synth.water_box(300, seed=72, L_A=20.8), synth.water_box(3000, seed=73), synth.silica_box(600, seed=74),
               synth.silica_box(4000, seed=75), synth.uniform_gas(1057, 24.0, seed=76, n_types=3),
               synth.uniform_gas(40, 30.0, seed=77, n_types=1)]
    box = epsr.Box(systems)
    H = torch.zeros((3, box.hist_len), dtype=torch.int64, device=DEV)
    box.epsr_partial_gr(H[0])
    box.epsr_partial_gr_cells(H[1])
    box.epsr_partial_gr_range(0, box.epsr_partial_gr_tiles(), H[2])
    assert torch.equal(H[0], H[2]) and torch.equal(H[1], H[2])
    h0 = 0
    for s in systems:
        ref = oracle.Box(s).histogram(threads=8)
        assert np.array_equal(H[0, h0:h0 + ref.size].cpu().numpy().astype(np.uint64).reshape(ref.shape), ref)
        h0 += ref.size


@pytest.mark.parametrize("near_all,r_lj,ctas", [(True, 0.0, 0), (True, 6.0, 3), (False, 6.0, 1), (False, 0.0, 1)],
                         ids=["near-all", "near-all-cut", "global-cut", "global"])
def test_sweep_paths_replay(near_all, r_lj, ctas):
    """Every chunk near, and slices in global memory (22,500 atoms on one CTA), with Lennard-Jones cut and not."""
    n_mol = 1500 if near_all else 15000
    s = mixed_box([1, 2], n_mol, 3, seed=31, n_bins=150, r_lj=r_lj)
    box = epsr.Box(s)
    if near_all:
        box.epsr_mc_set_cells(0, 0)
    if ctas:
        box.epsr_mc_set_ctas(ctas)
    _, log = run_logged(box, 500, seed=23)
    ob, _, _, flips = replay(s, s.xyz, log[0], 23)
    assert flips <= 2
    assert np.array_equal(box.epsr_box_get_coords(), ob.xyz)


@pytest.mark.parametrize("sizes,n_mol,ctas,r_lj,moves", [([1], 700, 0, 4.0, 6000), ([1], 700, 1, 0.0, 4000), ([2, 3], 250, 5, 0.0, 4000),
                                                         ([1], 3000, 0, 4.0, 6000)])
def test_large_steps_replay(sizes, n_mol, ctas, r_lj, moves):
    """Steps of 2 A in a dense box: trials land on top of molecules that an earlier move of the batch takes away,
    so a dU of a few kJ/mol is what is left of 10^4 and more. Every move against the oracle, with the bars of all replays."""
    s = mixed_box(sizes, n_mol, 2, seed=n_mol, n_bins=100, spacing=3.2, r_lj=r_lj)
    s.r_coul, s.eps, s.max_translation = 0.0, [0.4, 0.4], 2.0
    box = epsr.Box(s)
    if ctas:
        box.epsr_mc_set_ctas(ctas)
    _, log = run_logged(box, moves, seed=24)
    ob, _, _, flips = replay(s, s.xyz, log[0], 24)
    assert flips <= 2
    assert np.array_equal(box.epsr_box_get_coords(), ob.xyz)
