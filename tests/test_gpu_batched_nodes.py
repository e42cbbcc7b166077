"""Batches whose graph holds one single-view kernel per job (large float
views; sparse views of any storage type): every image and sample count equals
the single renders bit for bit, on the first launch and replayed, on two
streams at once, and after the batch ran without a graph."""
import pytest

import synth
from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _jobs(torch, P, store, sizes, dims_of):
    out = []
    for q, (w, h) in enumerate(sizes):
        dims = dims_of(q)
        vol = P.Volume(synth.hi_cube(dims, n_blobs=5, n_disks=0, seed=q).cuda(), store)
        tf = synth.tf_ramp(256) if q % 2 else synth.tf_random_pwl(seed=q)
        out.append(dict(vol=vol, cam=synth.camera_random_persp(dims, seed=20 + q, width=w, height=h),
                        tf=torch.from_numpy(tf).cuda(), vmin=-3.0, vmax=40.0, step=0.7, ert=0.99 if q % 3 else 2.0,
                        out=torch.empty((h, w, 4), device="cuda"),
                        nsamples=torch.empty((h, w), device="cuda", dtype=torch.int32)))
    return out


@pytest.mark.parametrize("store,sizes,dims_of", [
    ("f32", [(640, 450), (701, 502), (512, 515), (530, 700)], lambda q: (60 + 9 * q, 71, 50)),
    ("f32", [(20, 17), (31, 24), (1, 1)], lambda q: (150, 120 + q, 140)),
    ("f16", [(24, 19), (33, 30), (200, 170)], lambda q: (170, 150, 130 + q)),
    ("bf16", [(24, 19), (25, 31)], lambda q: (170, 150, 130 + q))], ids=["large", "sparse32", "sparse16", "sparseb16"])
def test_nodes_equal_single_renders(torch, store, sizes, dims_of):
    import paper_1211_4896_gb300 as P
    jobs = _jobs(torch, P, store, sizes, dims_of)
    try:
        ref = [P.render(j["vol"], j["cam"], j["tf"], j["vmin"], j["vmax"], j["step"], j["ert"]) for j in jobs]

        def check(which=jobs):
            torch.cuda.synchronize()
            for j, (img, ns) in zip(which, ref):
                assert torch.equal(j["out"], img) and torch.equal(j["nsamples"], ns)
                j["out"].fill_(-1.0)
                j["nsamples"].fill_(-1)
            torch.cuda.synchronize()

        for graph in (True, True, False, True):
            P.render_batched(jobs, use_graph=graph)
            check()
        jobs[0]["tf"].copy_(jobs[-1]["tf"])                 # the table is read at each launch
        ref[0] = P.render(jobs[0]["vol"], jobs[0]["cam"], jobs[0]["tf"], jobs[0]["vmin"], jobs[0]["vmax"],
                          jobs[0]["step"], jobs[0]["ert"])
        P.render_batched(jobs)
        check()
        other = [dict(j, out=torch.empty_like(j["out"]), nsamples=torch.empty_like(j["nsamples"])) for j in jobs]
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        for _ in range(3):                                   # a stream's plan has counters of its own
            P.render_batched(jobs)
            P.render_batched(other, stream=side)
        check()
        check(other)
    finally:
        for j in jobs:
            j["vol"].close()
