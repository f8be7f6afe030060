// paths.cuh -- arguments and launchers of dedupe, validation and reduction.
#pragma once

#include "dcem_internal.cuh"

namespace dcem {

struct PathArgs {
  int R;                          // segment-log stride (rays, plus child slots with transmission)
  const int* log_id;              // (N+1) x R hit ids
  const Cand* cand;
  unsigned cand_cap;
  unsigned long long* hkey;       // hash slots: 64-bit key, 0 = empty
  unsigned long long* hrep;       // (ray << 32 | candidate) of the representative, ~0 = none
  unsigned hcap;                  // power of two
  int* cand_slot;                 // per candidate
  int* uniq;                      // representative candidate per distinct key
  unsigned ucap;
  PathRec* prec;                  // per distinct key
  const int* ray_perm;            // ray slot -> caller's ray index
  double* vpts;                   // per distinct key: (kMaxRefl + 2) FP64 path points
  int* vstate;                    // per distinct key: 0 invalid, 1 valid so far, 2 occluded
  int N;                          // reflections (sub-segments per path <= N + max_trans + 1)
  int max_trans;                  // transmissions per path (ids with kTransBit)
  int R0;                         // primary rays; slots from R0 on are transmission children
  const int* inst_root;           // per child slot: its primary ray's slot
  int* bucket;                    // links x bucket_cap distinct-key indices of valid paths
  unsigned* bucket_cnt;           // links (link = transmitter * nrx + receiver)
  int bucket_cap;                 // power of two
  unsigned* link_off;             // groups of links: their paths, or their output offsets (many links); or null
  dcem_path* pout;                // ordered output (link, key): caller's device buffer or staging
  unsigned pout_cap;
  dcem_path* hrec;                // first hrec_cap records: mapped host memory in place of pout
  unsigned hrec_cap;
  double* out_field;              // links x 2 (re, im), or null
  double* out_pc;                 // links P_coh dBm, or null
  double* out_pi;                 // links P_inc dBm, or null
  const float4* tris;             // leaf-ordered triangles
  const int* slot_of_id;
  const float4* mats;             // eps_r, sigma, pec
  Bvh bvh;
  const float4* rx;               // nrx receivers
  int nrx;
  const float4* txs;              // per transmitter: position (xyz)
  float3 pol;
  float eps_occ;
  int prec_df;                    // 1: validation geometry in double-float, 0: FP64
  double freq, tx_power;
  DevCounters* ctr;
  // sticky mode (null otherwise): the previous frame's valid paths, to be
  // re-validated when no capture of this frame has their key, and the
  // buffer that keeps this frame's valid paths for the next one
  // first-order edge diffraction (null: off)
  Wedge* wedges;                  // geometry, rebuilt every frame from the world triangles
  WedgeF* wf;                     // the same in FP32 (pre-tests)
  const WedgeTopo* wtopo;
  int nw;
  // the wedges in a fixed spatial order (wperm): nwc mask words of
  // kWedgeCluster, and the boxes of the groups of kWedgeGroup (6 floats
  // each, every frame)
  const int* wperm;
  const int* wplace;              // ... and each wedge's place in it
  float* wgbox;
  int nwc;
  unsigned long long* dsurv;      // candidates past the FP32 pre-tests
  unsigned long long* dexact;     // ... and past the FP32 occlusion test (same capacity)
  unsigned dsurv_cap;
  // one reflection before or after a diffraction (null: off): reflector
  // planes and their member triangle ids
  const RPlane* rplanes;
  const int* rmembers;             // per plane its members, sorted by their lowest coordinate
  const float* rkeys;              // along the plane's axis, and that coordinate
  int nrp;
  const float4* quads;            // per triangle id: the convex wall quad it is part of (corners; .w of
                                  // the first 0: none)
  int open;                       // 1: an open scene, little of which is hidden (launch_hidden_planes)
  int rsub;                       // runs of receivers per transmitter item (set by launch_diffract)
  unsigned* vis;                  // per end point: bits of the planes, then of the wedges it may see
  unsigned* vis_any;              // the wedges some transmitter, then some receiver may see
  int* vis_grp;                   // ... and the groups that hold any: per side a count and the list
  int drefl2;                     // 1: also two reflections around a first-order diffraction
  unsigned* rmask;                // with drefl2: the wedge masks of k_refl_single, one word per
                                  // (end point: transmitters then receivers, plane, cluster)
  unsigned* wobs_cnt;             // with drefl2, per wedge: the receivers' one-reflection sides,
  unsigned* wobs_off;             // where they start in dobs, and the next free slot there
  unsigned* wobs_pos;
  DiffObs* dobs;
  unsigned dobs_cap;
  int dmid;                       // 1: also a reflection between the two wedges of an order-2 chain
  // diffraction of order 2 and 3 (diff_order <= 1: off): the wedge pairs
  // (v, w1, w2, -1), the pairs with a reflection on plane p between them
  // (t, w1, w2, -2 - p) and triples (v, w1, w2, w3) of the frame, v a source
  // (a transmitter, or with reflector planes the image of transmitter t in
  // plane p: v = dntx + t * nrpr + p), and the pair relation as a bit matrix
  // (nw x nw bits)
  int diff_order;
  int dntx;                       // transmitters (set by launch_diffract)
  int nrpr;                       // reflector planes applied to chains (0: none; set by launch_diffract)
  int4* dseq2;
  unsigned dseq2_cap;
  int4* dseq3;
  unsigned dseq3_cap;
  unsigned* drel;
  // order 3: the receivers past stage 1 at each related pair (null: the rows
  // would take too much memory, stage 1 is then run per triple), and the
  // wedges that are second in some pair (bits)
  unsigned* dobs1;
  int dobs1_row;
  unsigned* dsecond;
  // validation reuse (coherent frames; Sec. III "Propagation path caching"):
  // the previous frame's records of its distinct keys, found through a hash
  // table of their link keys, are copied when nothing they depend on moved
  int reuse;                      // 1: look the keys up in the previous frame's table
  const unsigned long long* vc_prev_key;  // previous table: link key (0 = empty) and record index
  const unsigned* vc_prev_u;
  const PathRec* prev_prec;       // the previous frame's records, points and states
  const double* prev_vpts;
  const int* prev_vstate;
  unsigned vc_cap;                // slots of each table (power of two)
  unsigned long long* vc_next_key;  // this frame's table (built after validation), or null
  unsigned* vc_next_u;
  unsigned long long* ckey;       // per distinct key of this frame: its link key
  const unsigned char* rx_moved;  // receivers whose position changed
  const unsigned char* obj_moved; // rigid objects whose transform changed
  const int* tri_obj;             // triangle id -> rigid object (-1 static)
  SmallBvh mvt;                   // the moved objects' old and new boxes
  unsigned mv_cap;                // boxes the tree holds (more moved boxes: no reuse)
  const StickyKey* sticky_prev;
  const unsigned* sticky_prev_n;
  unsigned sticky_cap;
  StickyKey* sticky_next;
};

cudaError_t launch_dedupe(const PathArgs& a, int grid, cudaStream_t st);
// Sticky mode: the previous frame's valid paths whose key no capture of this
// frame has join the distinct keys (validated like them).
cudaError_t launch_sticky_probe(const PathArgs& a, int grid, cudaStream_t st);
// Frames of at most kFewLinks links validate in one kernel, a group of lanes
// per key (a few hundred keys: latency); more links in three (tens of thousands
// of keys: throughput).
constexpr int kFewLinks = 1024;
cudaError_t launch_validate(const PathArgs& a, int nlinks, int grid, cudaStream_t st);
// The table of this frame's distinct keys for the next frame's validation
// reuse (after validation, before diffraction adds its records).
cudaError_t launch_vcache_build(const PathArgs& a, int grid, cudaStream_t st);
// How much of a scene its walls hide: of cnt[1] sampled pairs of reflector
// planes cnt[0] are hidden from each other (a: the static tree, quads, planes,
// eps_occ). Open scenes, with at most kOpenNum in kOpenDen of them, go without
// visibility and occlusion tests, and test both reflections on one side of a
// wedge link by link. Roads: 0 (barriers in one piece) to 30% (in twenty, each
// a little further out), 2 x 2 city blocks 30 and 33%, 3 x 3 44 and 47%, 4 x 4
// 55 and 58%, 8 x 8 76 and 78% (two seeds each), an urban grid 97%.
// us a frame, open / with tests, two reflections and chains of two with one:
// road in eight pieces 2706 / 5263 and 5142 / 5209, 2 x 2 355 / 426 and 344 /
// 435, 3 x 3 (60 receivers) 866 / 790 and 554 / 706, 5 x 5 1752 / 1158 and 880
// / 1026, 8 x 8 14456 / 2376 and 5594 / 3337.
constexpr unsigned kOpenNum = 3, kOpenDen = 8;
cudaError_t launch_hidden_planes(const PathArgs& a, unsigned* cnt, cudaStream_t st);
// First-order edge diffraction paths of every (link, wedge) (after validation).
cudaError_t launch_diffract(const PathArgs& a, int nlinks, int sms, cudaStream_t st);
// Per-link sums and ordered output; more links than kScanLinks take their
// output offsets from sums over groups (a.link_off) instead of summing the
// lower links' counts.
constexpr int kScanLinks = 4096;
cudaError_t launch_reduce(const PathArgs& a, int nlinks, cudaStream_t st);

}  // namespace dcem
