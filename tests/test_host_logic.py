"""Host side of the library without a GPU: which device memory belongs to, who waits for what, what happens when an
allocation fails.  Two pretended devices (tests/fake_cudart.cpp); kernels do not run, they only report sizes."""
import pytest

from tests import fake_device


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    return fake_device.build(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def fake(so):
    return fake_device.Fake(so)


def test_sizes_read_while_another_device_is_current(fake):
    """Sample on device 1, then on device 0, then ask for the sizes of the first object: what its context needs is made on
    device 1, and no block changes its device."""
    ctx1, ctx0 = fake.context(1), fake.context(0)
    fake.report(PHI=5000, PSI=6000, EDGES=900)
    rc, on1 = fake.sample(ctx1, 100)
    assert rc == 0
    rc, on0 = fake.sample(ctx0, 100)
    assert rc == 0
    live0 = fake.lib.fake_live(0)
    assert fake.lib.fake_current() == 0
    assert fake.nnz(on1) == (0, 5000) and fake.nnz(on1, 2) == (0, 6000)
    assert fake.lib.fake_live(0) == live0
    fake.report(EDGES=90000)                      # grows what was made above
    assert fake.sample(ctx1, 100, on1)[0] == 0
    fake.lib.fake_set_current(0)
    assert fake.nnz(on1)[0] == 0
    assert fake.sample(ctx0, 100, on0)[0] == 0
    assert fake.sample(ctx1, 100, on1)[0] == 0    # its launches find their memory on device 1
    assert fake.errors() == 0
    for h in (on0, on1):
        assert fake.lib.grf_features_free(h) == 0
    for c in (ctx0, ctx1):
        assert fake.lib.grf_ctx_destroy(c) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0 and fake.lib.fake_live(1) == 0


def test_reading_sizes_leaves_the_sampling_context_alone(fake):
    """One thread samples with its context while another, with its own context, takes the object on: whatever the second
    does to learn the sizes neither allocates nor waits for the device, and needs nothing of the first context."""
    ctx = fake.context(0)
    fake.report(PHI=5000, PSI=6000, EDGES=900)
    assert fake.lib.grf_ctx_destroy(fake.context(0)) == 0
    rc, a = fake.sample(ctx, 100)
    assert rc == 0
    fake.report(PHI=4000, PSI=3000, EDGES=1800)
    rc, b = fake.sample(ctx, 100)                 # the sizes of the first have not been read
    assert rc == 0
    mallocs, frees = fake.lib.fake_mallocs(), fake.lib.fake_frees()
    fake.lib.fake_log_clear()
    assert fake.nnz(a) == (0, 5000) and fake.nnz(a, 2) == (0, 6000)
    assert fake.log() in ([], ["sync event"])
    assert (mallocs, frees) == (fake.lib.fake_mallocs(), fake.lib.fake_frees())
    assert fake.lib.grf_ctx_destroy(ctx) == 0     # before the second object's sizes were read
    assert fake.nnz(b) == (0, 4000) and fake.nnz(b, 1) == (0, 3000)
    assert fake.lib.grf_features_free(a) == 0 and fake.lib.grf_features_free(b) == 0
    assert fake.errors() == 0


def test_a_sample_does_not_wait_for_the_one_before(fake):
    """... and the room for its edge records follows the graphs seen so far without a wait."""
    ctx = fake.context(0)
    fake.report(PHI=500, PSI=600, EDGES=900)
    rc, feat = fake.sample(ctx, 100)
    assert rc == 0 and fake.nnz(feat) == (0, 500)
    assert fake.sample(ctx, 100, feat)[0] == 0    # arrays are as large as they get
    fake.lib.fake_log_clear()
    fake.report(PHI=510, PSI=610)
    assert fake.sample(ctx, 100, feat)[0] == 0
    assert not [x for x in fake.log() if x.startswith("sync")]
    assert fake.nnz(feat) == (0, 510)
    assert fake.lib.grf_features_free(feat) == 0 and fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_an_object_whose_resampling_failed_is_empty(fake):
    """Not one with the new row count and the old, or no, arrays behind it."""
    ctx = fake.context(0)
    fake.report(PHI=5000, PSI=6000, EDGES=900)
    rc, feat = fake.sample(ctx, 100)
    assert rc == 0 and fake.nnz(feat) == (0, 5000)
    fake.lib.fake_limit(0, 300 << 20)             # the staging area fits, the matrices do not
    fake.report(PHI=40 << 20, PSI=40 << 20)
    assert fake.sample(ctx, 40000, feat)[0] == fake.NOMEM
    fake.lib.fake_log_clear()
    assert fake.linear(ctx, feat, 1, 40000, 32, 64, "fp32") == fake.INVALID
    assert fake.linear(ctx, feat, 1, 100, 32, 64, "fp32") == fake.INVALID
    assert fake.lib.grf_features_materialise(ctx, feat) != 0
    assert fake.launched("kernel") == 0 and fake.nnz(feat) == (0, 0)
    fake.lib.fake_limit(0, 1 << 40)
    fake.report(PHI=5000, PSI=6000)
    assert fake.sample(ctx, 100, feat)[0] == 0 and fake.nnz(feat) == (0, 5000)
    assert fake.linear(ctx, feat, 1, 100, 32, 64, "fp32") == 0
    assert fake.lib.grf_features_free(feat) == 0 and fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def _cloud_like(fake, ctx):
    """An object whose reported sizes are those of a cloud of 4096 points: the cost rule takes the mask."""
    fake.report(PHI=400_000, PSI=400_000, EDGES=40_000, PLAN=25_600, KEYS=64_000, POSITIONS=2_500_000, LONGEST=4096)
    rc, feat = fake.sample(ctx, 4096)
    assert rc == 0
    assert fake.lib.grf_plan_stats(ctx, feat, None, None) == 0
    return feat


def test_no_memory_for_the_mask_means_the_states(fake):
    """The main call does not fail for want of memory that the per-node states do without, and such a call does not keep
    grf_features_materialise from trying again."""
    ctx = fake.context(0)
    taken = {}
    for mib in (1, 2, 4, 6, 8, 12, 16, 20, 24, 32, 64):
        feat = _cloud_like(fake, ctx)
        fake.lib.fake_limit(0, fake.lib.fake_live(0) + (mib << 20))
        for _ in range(2):                        # the second call takes the same route
            fake.lib.fake_log_clear()
            assert fake.linear(ctx, feat, 8, 4096, 32, 64, "bf16") == 0, f"{mib} MiB left"
            mask, states = fake.launched("mhat_attention_kernel"), fake.launched("build_states")
            assert (mask > 0) != (states > 0)
            assert taken.setdefault(mib, mask > 0) == (mask > 0)
        fake.lib.fake_limit(0, 1 << 40)
        assert fake.lib.grf_features_materialise(ctx, feat) == 0
        assert fake.lib.grf_features_free(feat) == 0
        assert fake.lib.grf_ctx_destroy(ctx) == 0                 # gives the pool back
        ctx = fake.context(0)
    assert not taken[1] and taken[64] and len(set(taken.values())) == 2
    assert fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_pair_records_without_memory_or_with_the_callers(fake):
    """Records find room in the context's scratch; without memory for that, narrower ones in the workspace (two launches a problem
    instead of one, the same bits); whole states only where these do not fit either.  A workspace that holds all records means
    that no scratch is taken at all."""
    N, G, m, d = 20011, 3, 32, 64
    for nnz, narrow in ((1_200_000, True), (1_500_000, False)):
        ctx = fake.context(0)
        fake.report(PHI=nnz, PSI=nnz, EDGES=160_000)
        rc, feat = fake.sample(ctx, N)
        assert rc == 0
        live = fake.lib.fake_live(0)
        records = nnz * (d + 1) * 4 + 512
        fake.lib.fake_log_clear()
        assert fake.linear(ctx, feat, G, N, m, d, "fp32", workspace=G * records) == 0
        assert fake.launched("pair_records") == 1 and fake.lib.fake_live(0) == live
        fake.lib.fake_limit(0, live + (64 << 20))
        for _ in range(2):
            fake.lib.fake_log_clear()
            assert fake.linear(ctx, feat, G, N, m, d, "fp32") == 0
            assert fake.launched("pair_records") == (2 * G if narrow else 0)
            assert (fake.launched("build_states") == 0) == narrow
        fake.lib.fake_limit(0, 1 << 40)
        fake.lib.fake_log_clear()
        assert fake.linear(ctx, feat, G, N, m, d, "fp32") == 0
        assert fake.launched("pair_records") == G and fake.launched("build_states") == 0
        assert fake.lib.fake_live(0) - live <= (512 << 20) + (4 << 20)
        assert fake.lib.grf_features_free(feat) == 0 and fake.lib.grf_ctx_destroy(ctx) == 0
        assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_fp32_calls_that_wait_for_a_running_sample(fake):
    """Only one whose choice between records and whole states needs the sizes; none in the modes that keep to whole states."""
    ctx = fake.context(0)
    N, m, d = 4096, 32, 64
    fake.report(PHI=400_000, PSI=400_000, EDGES=40_000)
    rc, feat = fake.sample(ctx, N)
    assert rc == 0
    for mode, G, walks, waits in ((1, 3, 32, True), (2, 3, 32, True), (0, 3, 32, False), (3, 3, 32, False), (1, 1, 1, False)):
        assert fake.lib.grf_ctx_use_tensor_cores(ctx, mode) == 0
        for _ in range(2):                        # the second sample finds arrays that are large enough
            assert fake.sample(ctx, N, feat, walks=walks)[0] == 0
        fake.lib.fake_log_clear()
        assert fake.linear(ctx, feat, G, N, m, d, "fp32") == 0
        assert ("sync event" in fake.log()) == waits, (mode, G)
        assert (fake.launched("pair_records") > 0) == waits
    assert fake.lib.grf_features_free(feat) == 0 and fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_a_captured_call_without_room_for_denominators(fake):
    """Eager calls of its shape use the states where they are made and need none for a caller who asks for none.  The captured call
    finds its room all the same, and no later call takes that away from the graph."""
    A, B = (fake.lib.fake_stream(0) for _ in range(2))
    ctx, other = fake.context(0, A), fake.context(0, B)
    N, m, d = 4096, 32, 64
    fake.report(PHI=400_000, PSI=400_000, EDGES=40_000)
    rc, feat = fake.sample(ctx, N)
    assert rc == 0
    fake.lib.fake_log_clear()
    assert fake.linear(ctx, feat, 3, N, m, d, "fp32") == 0
    assert fake.launched("pair_records") > 0 and fake.launched("gather_denominators") == 0
    named, room = [], fake.lib.grf_attn_workspace_bytes(1, N, m, d, 0)
    for G in (3, 3, 4):                           # the last graph's block is another one than that of the first two
        fake.lib.fake_capture(A)
        assert fake.linear(ctx, feat, G, N, m, d, "fp32", workspace=G * room) == 0
        fake.lib.fake_capture(None)
        named.append(fake.lib.fake_denominators())
    assert fake.launched("pair_records") == 1 and fake.launched("gather_denominators") == 3
    assert named[0] == named[1] != named[2] and fake.errors() == 0
    assert fake.lib.grf_ctx_use_tensor_cores(ctx, 0) == 0 and fake.lib.grf_ctx_use_tensor_cores(other, 0) == 0
    for c in (ctx, other):                        # larger and equal calls
        for G in (3, 4, 6, 40):
            assert fake.linear(c, feat, G, N, m, d, "fp32", workspace=G * room) == 0
            if c is other or G == 40:
                assert fake.lib.fake_denominators() not in named
    assert fake.lib.grf_features_free(feat) == 0
    assert fake.lib.grf_ctx_destroy(ctx) == 0 and fake.lib.grf_ctx_destroy(other) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_a_captured_call_without_the_gathers_coefficients(fake):
    """Rows that share some of their nodes: eager calls use the states where they are made, a captured one gathers them by tiles.  The
    coefficients are built once, beside the graph."""
    A = fake.lib.fake_stream(0)
    ctx = fake.context(0, A)
    N, G, m, d = 20000, 8, 32, 64
    fake.report(PHI=500_000, PSI=500_000, EDGES=160_000, PLAN=78_000)
    rc, feat = fake.sample(ctx, N)
    assert rc == 0 and fake.lib.grf_ctx_use_tensor_cores(ctx, 2) == 0
    room = G * fake.lib.grf_attn_workspace_bytes(1, N, m, d, 1)
    assert fake.linear(ctx, feat, G, N, m, d, "bf16", workspace=room) == 0
    assert fake.launched("pair_records") > 0 and fake.launched("block_coef") == 0
    fake.lib.fake_log_clear()
    for _ in range(2):
        fake.lib.fake_capture(A)
        assert fake.linear(ctx, feat, G, N, m, d, "bf16", workspace=room) == 0
        fake.lib.fake_capture(None)
    assert fake.launched("gather_contract_tc") == 2 and fake.launched("pair_records") == 0
    assert [x for x in fake.log() if "block_coef" in x and x.endswith("beside")] and fake.launched("block_coef") == 1
    assert fake.lib.grf_features_free(feat) == 0 and fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_small_graphs_without_tensor_maps(fake):
    """The kernel for up to 512 nodes copies boxes through tensor maps, which the pretended driver does not make: the kernel that
    gathers rows takes the call."""
    ctx = fake.context(0)
    fake.report(PHI=40_000, PSI=40_000, EDGES=3200, PLAN=1600, KEYS=1664, POSITIONS=200_000, LONGEST=448)
    rc, feat = fake.sample(ctx, 400)
    assert rc == 0 and fake.lib.grf_features_materialise(ctx, feat) == 0
    some = fake_device.C.c_void_p(4096)
    for m in (16, 32, 64):
        fake.lib.fake_log_clear()
        assert fake.lib.grf_masked_attn_mhat(ctx, feat, 200, 400, m, 64, 1, some, some, some, some, None) == 0
        assert fake.launched("mhat_attention_kernel") == 1 and fake.launched("mhat_small_kernel") == 0
    assert fake.lib.grf_features_free(feat) == 0 and fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_host_path_without_memory_for_the_preferred_mask(fake):
    ctx = fake.context(0)
    fake.report(PHI=400_000, PSI=400_000, EDGES=8192, PLAN=25_600, KEYS=640_000, POSITIONS=2_500_000, LONGEST=40_000)
    assert fake.lib.grf_ctx_use_tensor_cores(ctx, 2) == 0
    for _ in range(2):                            # the second pass has made the object's arrays as large as they get
        assert fake.step_host(ctx, 4096, 8, 32, 64) == 0
    assert fake.lib.grf_ctx_prefer_mask_route(ctx, 1) == 0
    fake.lib.fake_limit(0, fake.lib.fake_live(0) + (1 << 20))
    fake.lib.fake_log_clear()
    assert fake.step_host(ctx, 4096, 8, 32, 64) == 0
    assert fake.launched("build_states") > 0 and fake.launched("mhat_attention_kernel") == 0
    fake.lib.fake_limit(0, 1 << 40)
    fake.lib.fake_log_clear()
    assert fake.step_host(ctx, 4096, 8, 32, 64) == 0
    assert fake.launched("build_states") == 0 and fake.launched("mhat_attention_kernel") > 0
    assert fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_host_path_that_fails_waits_for_its_copies(fake):
    """The caller may free or change its buffers once the call has returned, with an error as well."""
    ctx = fake.context(0)
    fake.report(PHI=5000, PSI=6000, EDGES=800)
    fake.lib.fake_log_clear()
    assert fake.step_host(ctx, 400, 8, 32, 64, walks=0) == fake.INVALID
    waited = {x for x in fake.log() if x.startswith("sync stream")}
    assert len(waited) >= 2                       # the context's stream and the one that the inputs travel on
    assert fake.step_host(ctx, 400, 8, 32, 64) == 0
    assert fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_objects_sampled_once_hold_what_their_entries_need(fake):
    """A model freezes one object per layer and head: its arrays follow the number of non-zeros.  An object that is sampled
    again and again has arrays for the largest sample, and its samples do not wait."""
    ctx = fake.context(0)
    nnz = 400_000
    fake.report(PHI=nnz, PSI=nnz, EDGES=40_000)
    rc, first = fake.sample(ctx, 4096)            # makes the context's scratch
    assert rc == 0
    live = fake.lib.fake_live(0)
    rc, frozen = fake.sample(ctx, 4096)
    assert rc == 0 and fake.nnz(frozen) == (0, nnz)
    assert fake.lib.fake_live(0) - live < 1.3 * 3 * (8 * nnz + 4 * 4097)
    for _ in range(2):
        assert fake.sample(ctx, 4096, first)[0] == 0
    fake.lib.fake_log_clear()
    assert fake.sample(ctx, 4096, first)[0] == 0
    assert not [x for x in fake.log() if x.startswith("sync")]
    for h in (first, frozen):
        assert fake.lib.grf_features_free(h) == 0
    assert fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_no_exception_leaves_the_library_when_the_heap_is_exhausted(fake):
    """Bookkeeping that finds no host memory is left out: blocks go back to the device at once, times are not taken."""
    ctx = fake.context(0)
    fake.report(PHI=5000, PSI=6000, EDGES=900)
    rc, feat = fake.sample(ctx, 100)
    assert rc == 0 and fake.lib.grf_ctx_enable_timing(ctx, 1) == 0
    assert fake.sample(ctx, 100, feat)[0] == 0
    frees = fake.lib.fake_frees()
    fake.lib.fake_no_heap(1)
    assert fake.sample(ctx, 100, feat)[0] == 0
    ms, n = (fake_device.C.c_float * 10)(), (fake_device.C.c_int64 * 10)()
    assert fake.lib.grf_ctx_kernel_times(ctx, ms, n) == 0
    assert fake.lib.grf_features_free(feat) == 0
    assert fake.sample(ctx, 100)[0] == fake.NOMEM
    fake.lib.fake_no_heap(0)
    assert fake.lib.fake_frees() - frees >= 9     # three matrices of three arrays
    assert fake.lib.grf_ctx_destroy(ctx) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_what_one_context_builds_inside_an_object_another_waits_for(fake):
    """The first attention call forms the mask (or the gather's coefficients) on its own stream; the caller, who passes a
    const object, cannot know of it.  A call of another context lets its stream wait for that."""
    A, B = (fake.lib.fake_stream(0) for _ in range(2))
    a, b = fake.context(0, A), fake.context(0, B)
    wait = f"wait stream {hex(B)}"
    for m, kernel in ((32, "mask_values"), (128, "block_coef")):
        feat = _cloud_like(fake, a) if m == 32 else fake.sample(a, 4096)[1]
        fake.lib.fake_log_clear()
        assert fake.linear(a, feat, 8, 4096, m, 64, "bf16") == 0
        assert fake.launched(kernel) == 1 and not [x for x in fake.log() if x.startswith("wait")]
        assert fake.linear(a, feat, 8, 4096, m, 64, "bf16") == 0
        assert not [x for x in fake.log() if x.startswith("wait")]        # its own stream is in order
        fake.lib.fake_log_clear()
        assert fake.linear(b, feat, 8, 4096, m, 64, "bf16") == 0
        assert fake.log()[0] == wait
        if m == 32:
            assert fake.lib.grf_features_materialise(a, feat) == 0
            fake.lib.fake_log_clear()
            some = fake_device.C.c_void_p(4096)
            assert fake.lib.grf_masked_attn_mhat(b, feat, 8, 4096, m, 64, 1, some, some, some, some, None) == 0
            assert fake.lib.grf_mask_rows(b, feat, 1, some, some) == 0
            assert fake.log()[0] == wait and fake.log()[2] == wait
        assert fake.lib.grf_features_free(feat) == 0
    assert fake.lib.grf_ctx_destroy(a) == 0 and fake.lib.grf_ctx_destroy(b) == 0
    assert fake.errors() == 0 and fake.lib.fake_live(0) == 0


def test_the_pool_holds_at_most_one_gib_and_goes_with_the_last_context(fake):
    ctx, other = fake.context(0), fake.context(1)
    fake.report(PHI=12 << 20, PSI=12 << 20, EDGES=900)
    feats = [fake.sample(ctx, 100) for _ in range(6)]             # 0.3 GiB of matrices each
    assert all(rc == 0 for rc, _ in feats) and fake.lib.fake_live(0) > 3 << 29
    before = fake.lib.fake_live(0)
    for _, h in feats:
        assert fake.lib.grf_features_free(h) == 0
    left = fake.lib.fake_live(0)
    assert before - left > 1 << 29                # more than the pool takes has gone back to the device
    mallocs = fake.lib.fake_mallocs()
    rc, h = fake.sample(ctx, 100)                 # served by blocks of the freed objects
    assert rc == 0 and fake.lib.fake_mallocs() == mallocs and fake.lib.fake_live(0) == left
    fake.lib.fake_limit(0, left)                  # an allocation that fails empties the pool and tries again
    fake.report(PHI=18 << 20, PSI=18 << 20)
    rc, big = fake.sample(ctx, 100)
    assert rc == 0 and fake.lib.fake_refused() > 0
    for x in (h, big):
        assert fake.lib.grf_features_free(x) == 0
    assert fake.lib.grf_ctx_destroy(ctx) == 0 and fake.lib.fake_live(0) <= (1 << 30) + (1 << 20)
    assert fake.lib.grf_ctx_destroy(other) == 0 and fake.lib.fake_live(0) == 0 and fake.lib.fake_live(1) == 0
    assert fake.errors() == 0
