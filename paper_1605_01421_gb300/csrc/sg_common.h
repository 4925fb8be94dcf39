// sg_common.h -- internal types shared by the host runtime and the kernels of
// the SimInf GB300 engine.  Not part of the public ABI (include/siminf_gpu.h).
#pragma once

#include <stdint.h>

#include "siminf_gpu.h"

#define SG_MAX_GDATA 32

// Counter-stream identifiers: the fourth Philox counter word is
// (stream << 24) | replicate, so replicates, SSA draws and event draws never
// share a counter.
#define SG_STREAM_SSA 0u
#define SG_STREAM_EVENTS 1u
#define SG_STREAM_EMU 2u
#define SG_STREAM_AEM 3u

// Model tables in the layout the kernels read (passed by value).
struct SgTables {
  int32_t kind, n_nodes, n_comp, n_trans, n_v, n_ldata, n_select, n_shift;
  int8_t S[SG_MAX_TRANS][SG_MAX_COMP];   // S[j][p]: change of p by transition j
  uint32_t dep[SG_MAX_TRANS];            // bit k: recompute rate k after j
  uint32_t Emask[SG_MAX_SELECT];         // bit p: compartment p in E[, s]
  int8_t Nsh[SG_MAX_SHIFT][SG_MAX_COMP]; // Nsh[q][p] = N[p, q]
  double gdata[SG_MAX_GDATA];
  float g_lo[SG_MAX_GDATA], g_hi[SG_MAX_GDATA];  // FP32 neighbours: g_lo <= gdata <= g_hi
};

// A scheduled event in planned order, one 32-byte sector (two 16-byte loads;
// as eight arrays each event touched eight sectors).  An E1 event (exit,
// enter, internal transfer) is found through its node's list, so its node
// and dest fields hold what the walk along that list needs instead.
struct SgEvent {
  union {
    int32_t node;
    int32_t next;  // E1: day index of the node's next E1 event, or SG_NO_DAY
  };
  int32_t dest;    // E1: unused
  int32_t n;
  int8_t type;
  uint8_t select;
  int8_t shift;    // -1 = no shift
  uint8_t pad;
  double proportion;
  int64_t index;   // position in the caller's list (random stream key)
};
#define SG_NO_DAY 0x7fffffff

// Error word written by kernels: the first error wins (atomicCAS on code).
struct SgDevError {
  int32_t code;
  int32_t rep;
  int32_t node;
  int32_t day;
  long long event;
};

struct SgCounters {
  unsigned long long reactions;
  unsigned long long draws;
  unsigned long long events;
  unsigned long long rated;  // node-days whose rates were evaluated (sparse schedule)
};
