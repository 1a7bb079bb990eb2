// Block-table stage kernels of the request loop: one launch per RK stage over
// all member cases of a group (the dual-time pseudo-stage form is in
// dual32.cu, beside the single-case dual-time launch that shares it).  Kept in a module of their own: linked into the
// single-case module, these kernels slowed the replay of single-case step
// graphs by ~10% on GB300 (measured; kernel durations themselves unchanged).
#include "stage32.cuh"

namespace ibm {

// All entries of a stage in one launch: the body-tile entries of every member
// first (they carry the node rebuilds), then the plain-tile entries; blocks
// walk the combined table with a grid stride, so a grid smaller than the
// table makes the launch persistent.  Per entry the block runs the per-tile
// code of the case the entry falls in (the same source as the single-case
// kernels; compiled separately, so FP32 roundings may differ between them).
// Launched with programmatic dependent launch, its blocks are resident while
// the previous stage's last blocks finish (they wait at the top for it to
// complete).
// TVD / QUAD: the TVD-2 reconstruction and / or the quadratic IB / ghost reconstruction compiled in (a group
// holds cases of one variant)
// BLOCKS of NT threads per SM: BATCH_BLOCKS, BATCH_FEW (80 registers and 68 to 308 bytes of spills where 64 registers
// leave 152 to 384: a case's constants come from memory, not as operands from the parameters) or WIDE_BLOCKS
template <int STAGE, bool TVD, bool QUAD, int NT, int BLOCKS>
__global__ void __launch_bounds__(NT, BLOCKS) k_stage_f32_batch_one(const __grid_constant__ StageBatch b) {
  __shared__ TileSmem sm;
  __shared__ StageCase sc;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int nbody = b.body_start[b.n], total = nbody + b.plain_start[b.n];
  for (int e = blockIdx.x; e < total; e += gridDim.x) {
    const bool body = e < nbody;
    const int *start = body ? b.body_start : b.plain_start;
    const int ee = body ? e : e - nbody;
    int q = 0;
    while (q + 1 < b.n && start[q + 1] <= ee) q++;
    load_case<NT>(sc, b.cs[q]);
    const float *In = STAGE == 1 ? sc.M : (STAGE == 2 ? sc.F1 : sc.F2);
    float *Out = STAGE == 1 ? sc.F1 : (STAGE == 2 ? sc.F2 : nullptr);
    if (body)
      stage_tile<STAGE, true, false, false, false, TVD, QUAD, NT>(sc.k, sc.c, sc.M, In, Out, sc.D, sc.tag, sc.sid, sc.rs,
                                                              sc.tile_body, sc.body_tiles, sc.ds, sc.fuse_cfl != 0,
                                                              sc.ncfl, ee - start[q], sm, DualPtrs{}, nullptr,
                                                              sc.rsq);
    else
      stage_tile<STAGE, false, false, false, false, TVD, QUAD, NT>(sc.k, sc.c, sc.M, In, Out, sc.D, sc.tag, sc.sid,
                                                               sc.rs, sc.tile_body, sc.body_tiles, sc.ds,
                                                               sc.fuse_cfl != 0, sc.ncfl, ee - start[q], sm,
                                                               DualPtrs{}, nullptr, sc.rsq);
    __syncthreads();  // shared memory is reused by the next entry
  }
}

static bool table_wide(const StageBatch &b) {
  bool rebuild = false;
  for (int q = 0; q < b.n; q++) rebuild |= b.cs[q].nb > 0 && !b.cs[q].k.ib_advance;
  return stage_wide(b.plain_start[b.n], b.body_start[b.n], rebuild, b.cs[0].k.beside);
}

// Blocks of 128 threads per SM of a table of nt plain tiles.  Where the table is a wave or two, the spills lengthen
// every tile's chain and the eighth block is not needed; more tiles use the room.  Per step, eight blocks against six
// (the step before the packed tile in brackets): 640 x 512 alone 78 us, 68 (66), three of 384 x 384 88, 79 (81),
// 1024 x 512 96, 93 (91), moving 169, 160 (160), three of 512 x 512 136, 135 (130); 2048 x 1024 295, 307 (314).
extern "C" int ibm__batch_blocks(int nt, int sms) { return nt <= 20LL * sms ? BATCH_FEW : BATCH_BLOCKS; }

// Form of a table's launch: 0 BATCH_BLOCKS, 1 wide blocks, 2 BATCH_FEW.
static int table_form(const StageBatch &b) {
  const int nt = b.plain_start[b.n];
  if (table_wide(b)) return 1;
  return ibm__batch_blocks(nt, sm_count()) == BATCH_FEW && !crowded(nt, b.cs[0].k.beside) ? 2 : 0;
}

// Blocks of that form's stage kernel resident per SM.
extern "C" int ibm__batch_blocks_per_sm(int form, int tvd, int quad) {
  int per = 0;
#define IBM_OCC_N(T, Q, N, B) \
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_stage_f32_batch_one<1, T, Q, N, B>, N, 0)
#define IBM_OCC(T, Q)                                 \
  (form == 1   ? IBM_OCC_N(T, Q, WIDE, WIDE_BLOCKS)   \
   : form == 2 ? IBM_OCC_N(T, Q, NTH, BATCH_FEW)      \
               : IBM_OCC_N(T, Q, NTH, BATCH_BLOCKS))
  const cudaError_t e = tvd ? (quad ? IBM_OCC(true, true) : IBM_OCC(true, false))
                            : (quad ? IBM_OCC(false, true) : IBM_OCC(false, false));
#undef IBM_OCC
#undef IBM_OCC_N
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess ? per : 0;
}

int batch_stage_blocks(const StageBatch &b) {
  return ibm__batch_blocks_per_sm(table_form(b), b.cs[0].k.tvd2, b.cs[0].k.quad);
}

cudaError_t launch_stage_f32_batch_one(const StageBatch &b, int stage, int grid, bool pdl, cudaStream_t s) {
  const int total = b.body_start[b.n] + b.plain_start[b.n];
  if (total == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned int)(grid > 0 && grid < total ? grid : total));
  const int form = table_form(b);
  cfg.blockDim = dim3(form == 1 ? WIDE : NTH);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  const bool tvd = b.cs[0].k.tvd2 != 0, quad = b.cs[0].k.quad != 0;
  if (quad)
    for (int q = 0; q < b.n; q++)
      if (!b.cs[q].rsq) return cudaErrorInvalidValue;  // the quadratic kernels read the second probes
#define IBM_BATCH_N(S, T, Q, N, B) cudaLaunchKernelEx(&cfg, k_stage_f32_batch_one<S, T, Q, N, B>, b)
#define IBM_BATCH(S, T, Q)                              \
  (form == 1   ? IBM_BATCH_N(S, T, Q, WIDE, WIDE_BLOCKS) \
   : form == 2 ? IBM_BATCH_N(S, T, Q, NTH, BATCH_FEW)    \
               : IBM_BATCH_N(S, T, Q, NTH, BATCH_BLOCKS))
#define IBM_BATCH_S(S)                                                                                          \
  (tvd ? (quad ? IBM_BATCH(S, true, true) : IBM_BATCH(S, true, false))                                          \
       : (quad ? IBM_BATCH(S, false, true) : IBM_BATCH(S, false, false)))
  const cudaError_t e = stage == 1 ? IBM_BATCH_S(1) : stage == 2 ? IBM_BATCH_S(2) : IBM_BATCH_S(3);
#undef IBM_BATCH_S
#undef IBM_BATCH
#undef IBM_BATCH_N
  return e;
}

void build_stage_batch(const StageCase *cases, int n, StageBatch *b) {
  b->n = n;
  b->plain_start[0] = b->body_start[0] = 0;
  for (int q = 0; q < n; q++) {
    b->cs[q] = cases[q];
    b->plain_start[q + 1] = b->plain_start[q] + cases[q].nt;
    b->body_start[q + 1] = b->body_start[q] + cases[q].nb;
  }
}

void fill_stage_case(const Consts &k, float *M, float *F1, float *F2, double *D, const uint8_t *tag, const int *sid,
                     const RStencil32 *rs, const uint8_t *tile_body, const int *body_tiles, int body_cap,
                     DevState *ds, bool fuse_cfl, StageCase *out) {
  out->k = k;
  out->c = pert_consts(k);
  out->M = M;
  out->F1 = F1;
  out->F2 = F2;
  out->D = D;
  out->tag = tag;
  out->sid = sid;
  out->rs = rs;
  out->tile_body = tile_body;
  out->body_tiles = body_tiles;
  out->ds = ds;
  out->nt = stage_tiles(k);
  out->nb = body_cap > 0 ? body_cap : 0;
  out->fuse_cfl = fuse_cfl ? 1 : 0;
  out->ncfl = (unsigned int)(out->nt + out->nb);
  out->B = out->C = out->Q0 = nullptr;
  out->G = nullptr;
  out->rsq = nullptr;
}


}  // namespace ibm
